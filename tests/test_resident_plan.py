"""The cut of small lattices and batches into one rectangle per SM
(csrc/resident.cu), host code compiled here with g++ against stand-ins for the
few CUDA calls it makes: 152 SMs, and an operator new that can fail."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1611_00907_gb300 import _lib

CSRC = os.path.join(os.path.dirname(os.path.abspath(_lib.__file__)), "csrc")
MAIN = r"""
#include "resident.cu"
#include <cstdio>
#include <cstdlib>
static int g_fail = -1;
void *operator new(size_t n)
{
    if (g_fail >= 0 && g_fail-- == 0) throw std::bad_alloc();
    return malloc(n);
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
extern "C" {
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
namespace cplbm {
cudaError_t launch_resident_f64(const ResidentArgs &, bool, int, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_resident_f32(const ResidentArgs &, bool, int, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_resident_f32off(const ResidentArgs &, bool, int, int, size_t, cudaStream_t) { return cudaSuccess; }
bool current_context_id(unsigned long long *) { return false; }
}
// lines "failing precision count nx ny walls ..." -> "ok threads smem tiles: inst x0 y0 w h ..."
int main()
{
    int fail, prec, count;
    while (scanf("%d %d %d", &fail, &prec, &count) == 3) {
        std::vector<cplbm::Lattice> L(count);
        for (auto &l : L) {
            int walls;
            if (scanf("%d %d %d", &l.nx, &l.ny, &walls) != 3) return 1;
            l.walls = walls;
            l.nyf = walls ? l.ny - 2 : l.ny;
            l.precision = prec;
        }
        cplbm::ResidentPlan p;
        g_fail = fail;
        const bool ok = cplbm::resident_plan(L.data(), count, 0, &p);
        g_fail = -1;
        printf("%d %d %zu", ok, p.threads, p.smem);
        for (auto &t : p.tiles) printf(" %d %d %d %d %d", t.inst, t.x0, t.y0, t.w, t.h);
        printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    d = tmp_path_factory.mktemp("plan")
    (d / "main.cc").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, "-I" + cuda, "-x", "c++",
                    str(d / "main.cc"), "-o", str(d / "plan")], check=True)

    def run(lattices, prec=0, fail=-1):
        text = "%d %d %d " % (fail, prec, len(lattices))
        text += " ".join("%d %d %d" % (nx, ny, int(w)) for nx, ny, w in lattices)
        v = subprocess.run([str(d / "plan")], input=text, capture_output=True, text=True,
                           check=True).stdout.split()
        return bool(int(v[0])), int(v[1]), int(v[2]), np.array(v[3:], dtype=int).reshape(-1, 5)

    return run


# one tile; tiles of a few nodes; more than 256 nodes a tile (the 384- and
# 512-thread kernels) with odd and ragged sides; the largest that fit; batches
CASES = [
    [(5, 5, False)], [(7, 9, True)], [(64, 64, False)], [(250, 120, True)],
    [(331, 173, False)], [(331, 173, True)], [(500, 201, True)], [(5, 3001, False)],
    [(20001, 7, True)], [(521, 517, False)], [(519, 511, True)],
    [(70, 21, False), (33, 40, True), (64, 64, False)],
    [(32, 256, False)] * 28, [(131, 97, True)] * 8, [(40, 40, False)] * 152,
]


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_the_tiles_cover_every_lattice_once_and_fit(plan, case, prec):
    lats = CASES[case]
    ok, threads, smem, tiles = plan(lats, prec)
    if lats == [(20001, 7, True)] and prec == 0:
        # 152 tiles of 132 x 5 have 880 rim nodes each, 384 threads take 768
        assert not ok and len(tiles) == 0
        return
    assert ok and len(tiles) <= 152 and smem <= 220 * 1024
    assert threads in (256, 384 if prec == 0 else 512)
    for i, (nx, ny, walls) in enumerate(lats):
        nyf = ny - 2 if walls else ny
        seen = np.zeros((nyf, nx), dtype=int)
        for _, x0, y0, w, h in tiles[tiles[:, 0] == i]:
            assert w >= 1 and h >= 1 and x0 + w <= nx and y0 + h <= nyf
            # the rim nodes of a tile: two for each thread at most
            side = 4 if walls else 3
            assert 6 * (w + 2 * side) + 2 * side * h <= 2 * threads
            assert not (walls and h == 1)      # the solid row's density is the tile's own
            seen[y0:y0 + h, x0:x0 + w] += 1
        assert (seen == 1).all()


@pytest.mark.parametrize("lats,prec", [([(5000, 5000, False)], 0), ([(1024, 1024, False)], 1),
                                       ([(64, 64, False)], 3), ([(16, 16, False)] * 153, 1)])
def test_too_large_too_many_or_fp16_have_no_plan(plan, lats, prec):
    ok, _, _, tiles = plan(lats, prec)
    assert not ok and len(tiles) == 0


@pytest.mark.parametrize("lats", [[(64, 64, False)], [(70, 21, False), (33, 40, True)]])
def test_no_exception_leaves_it(plan, lats):
    """Every allocation it makes fails in turn: no plan, no exception."""
    ok, failed = False, 0
    while not ok:
        ok, _, _, tiles = plan(lats, 0, failed)
        assert ok or len(tiles) == 0
        failed += 1
        assert failed < 1000
    assert failed > 1
