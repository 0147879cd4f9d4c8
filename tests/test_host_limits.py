"""Host-side limits and sizes that keep kernels inside their buffers (no GPU)."""
import os
import random
import subprocess

from paper_2009_13507_gb300 import build as B

NACC = 11  # partial sums a block of the observables kernel writes

# prints the scratch's size, the scalars' slot and the accepted number of 32 x 4 blocks, then the
# observables kernel's grid for each "dim nx ny" of the input
PROBE = r"""
#include <stdio.h>
#include "sgpe_launch.h"
int main() {
    printf("%zu %zu %zu\n", sgpe::kObsScratchBytes, sgpe::kObsScalarsBytes, sgpe::kObsMaxBlocks);
    int dim, nx, ny;
    while (scanf("%d %d %d", &dim, &nx, &ny) == 3) {
        const dim3 g = sgpe::obs_grid(dim, nx, ny);
        printf("%u\n", g.x * g.y * g.z);
    }
}
"""


def test_static_observables_scratch_holds_every_accepted_grid(tmp_path):
    """sgpe_observables_noalloc accepts grids of up to kObsMaxBlocks blocks of 32 x 4 points; what the
    kernel launches writes NACC doubles a block behind the scalars' slot. Grids of three or four
    rows launch as many blocks as are counted: the last three column blocks used to end past the array."""
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    limit = 11912  # the documented bound of include/sgpe.h
    rng = random.Random(1)
    grids = [(2, 32 * b - q, ny) for b in range(limit - 4, limit + 1) for q in (0, 31) for ny in (3, 4)]
    grids += [(1, 32 * b - q, 1) for b in (1, 2, limit - 1, limit) for q in (0, 29)]
    grids += [(2, 3, 4 * limit), (2, 32, 4 * limit - 3)]
    for _ in range(500):
        cols = int(limit ** rng.random())
        rows = max(1, int((limit // cols) * rng.random()))
        grids.append((2, 32 * cols - rng.randrange(29), max(3, 4 * rows - rng.randrange(4))))
    out = subprocess.run([str(exe)], input="\n".join("%d %d %d" % g for g in grids), text=True, capture_output=True,
                         check=True).stdout.split()
    scratch, slot, accepted = (int(v) for v in out[:3])
    assert accepted == limit
    for (dim, nx, ny), blocks in zip(grids, map(int, out[3:])):
        counted = -(-nx // 32) * -(-ny // 4)
        assert counted <= limit and blocks <= counted, (dim, nx, ny)
        assert slot + blocks * NACC * 8 <= scratch, (dim, nx, ny, blocks)


def test_a_batch_is_created_and_sized_without_a_gpu():
    """sgpe_batch_create, _sizes and _offsets are host work: a caller can plan its buffers where no
    GPU is (the batch's streams are made when it is bound)."""
    import ctypes

    from paper_2009_13507_gb300 import sgpe
    lib = sgpe.load()
    inst = (sgpe.Instance * 2)()
    for i, (dim, nx, ny) in enumerate(((1, 128, 1), (2, 131, 140))):
        inst[i].dim, inst[i].nx, inst[i].ny, inst[i].dx, inst[i].dy = dim, nx, ny, 0.1, 0.1
        inst[i].params = sgpe.Physics(c0=1.0, dt=1e-3).c()
    b = ctypes.c_void_p()
    assert lib.sgpe_batch_create(ctypes.byref(b), 2, inst, sgpe.C64, None) == sgpe.OK
    elems, nbytes, offs = ctypes.c_size_t(), ctypes.c_size_t(), (ctypes.c_size_t * 2)()
    assert lib.sgpe_batch_sizes(b, ctypes.byref(elems), ctypes.byref(nbytes)) == sgpe.OK
    assert lib.sgpe_batch_offsets(b, offs) == sgpe.OK
    assert elems.value >= 3 * 128 + 3 * 131 * 140 and nbytes.value > 0 and offs[0] == 0 and offs[1] >= 3 * 128
    assert lib.sgpe_batch_destroy(b) == sgpe.OK
