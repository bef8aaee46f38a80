"""The dense inverses of the multigrid's coarsest operators by band elimination on the device
(csrc/vip_mg.cu), called through a small harness, against numpy's inverse of the same matrix:
lattices numbered along either side, periodic sides (also so short that couplings coincide),
single rows, empty cells, matrices that need row exchanges, and several sizes in one call.

Bar: Gaussian elimination with partial pivoting has a forward error below n eps times the
condition number times the growth factor; n <= 2200 and a growth of 4 give 1e-12 cond(A).
"""
import ctypes as C
import importlib
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HARNESS = r'''
#include "vip_mg.cu"
namespace vip { vip_status fail(vip_ctx*, vip_status s, const char*) { return s; } }
extern "C" int run(int G, int64_t ncell, const int* nx, const int* ny, const int64_t* c0, const double* coef,
                   const int* nbr, int64_t total, double* inv, float* inv32) {
    using namespace vip;
    vip_ctx c;
    Multigrid M;
    MgLevel lc;
    lc.n = ncell;
    cudaMalloc(&lc.coef, 25 * ncell * 8); cudaMalloc(&lc.nbr, 25 * ncell * 4);
    cudaMalloc(&M.cinv, total * 8); cudaMalloc(&M.cinv32, total * 4);
    cudaMemcpy(lc.coef, coef, 25 * ncell * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(lc.nbr, nbr, 25 * ncell * 4, cudaMemcpyHostToDevice);
    std::vector<BandMat> mats;
    std::vector<int2> dims;
    int64_t o = 0;
    for (int g = 0; g < G; ++g) {
        const int m = nx[g] * ny[g];
        mats.push_back({0, 0, o, c0[g], 0, m, 0, 0});
        dims.push_back(make_int2(nx[g], ny[g]));
        o += (int64_t)m * m;
    }
    int s = band_inverses(&c, M, lc, mats, dims, nbr);
    if (cudaMemcpy(inv, M.cinv, total * 8, cudaMemcpyDeviceToHost) != cudaSuccess) s = -1;
    cudaMemcpy(inv32, M.cinv32, total * 4, cudaMemcpyDeviceToHost);
    cudaFree(lc.coef); cudaFree(lc.nbr); cudaFree(M.cinv); cudaFree(M.cinv32);
    return s;
}
'''


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    build = importlib.import_module("paper_1401_6513_gb300.build")
    d = tmp_path_factory.mktemp("band")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS, *build.ARCH, "-w", "-I", str(build.CSRC), "-shared", str(d / "h.cu"),
                    "-o", str(d / "h.so")], check=True)
    return C.CDLL(str(d / "h.so"))


def lattice(nx, ny, px, py, dominant, rng):
    """coef, nbr [25][m] of a random 5 x 5 stencil; one cell in nine is empty and uncoupled."""
    m = nx * ny
    cell = np.arange(m)
    x, y = cell % nx, cell // nx
    empty = rng.random(m) < 1 / 9
    coef, nbr = np.zeros((25, m)), np.full((25, m), -1, np.int32)
    for o in range(25):
        xx, yy = x + o % 5 - 2, y + o // 5 - 2
        ok = np.ones(m, bool)
        xx, ok = (xx % nx, ok) if px else (xx, ok & (xx >= 0) & (xx < nx))
        yy, ok = (yy % ny, ok) if py else (yy, ok & (yy >= 0) & (yy < ny))
        nbr[o, ok] = (yy * nx + xx)[ok]
        live = ok & ~empty & ~empty[np.where(ok, nbr[o], 0)]
        coef[o, live] = rng.uniform(-1, 1, m)[live]
    if dominant:
        coef[12, ~empty] = 25.0
    return coef, nbr


CASES = [[(9, 8, 0, 0)], [(65, 33, 0, 0)], [(33, 65, 0, 0)], [(24, 40, 0, 1)], [(40, 24, 0, 1)], [(24, 40, 1, 0)],
         [(3, 40, 1, 0)], [(72, 1, 0, 0)], [(1, 72, 0, 0)], [(13, 12, 1, 1)],
         [(20, 17, 0, 0), (9, 9, 1, 0), (7, 31, 0, 1)]]


@pytest.mark.parametrize("dominant", [True, False])
@pytest.mark.parametrize("geoms", CASES, ids=str)
def test_band_inverse_matches_numpy(harness, geoms, dominant):
    rng = np.random.default_rng(11)
    parts = [lattice(*g, dominant, rng) for g in geoms]
    pad = [-p[0].shape[1] % 32 for p in parts]
    c0 = np.concatenate([[0], np.cumsum([p[0].shape[1] + q for p, q in zip(parts, pad)])]).astype(np.int64)
    coef = np.concatenate([np.pad(p[0], ((0, 0), (0, q))) for p, q in zip(parts, pad)], 1)
    nbr = np.concatenate([np.pad(np.where(p[1] >= 0, p[1] + c, -1), ((0, 0), (0, q)), constant_values=-1)
                          for p, q, c in zip(parts, pad, c0)], 1).astype(np.int32)
    sizes = [p[0].shape[1] for p in parts]
    total = sum(m * m for m in sizes)
    inv, inv32 = np.empty(total), np.empty(total, np.float32)
    nx, ny = (np.array([g[i] for g in geoms], np.int32) for i in (0, 1))
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    coef, nbr = np.ascontiguousarray(coef), np.ascontiguousarray(nbr)
    assert harness.run(len(geoms), C.c_int64(coef.shape[1]), ptr(nx), ptr(ny), ptr(c0), ptr(coef), ptr(nbr),
                       C.c_int64(total), ptr(inv), ptr(inv32)) == 0
    o = 0
    for (cf, nb), m in zip(parts, sizes):
        A = np.zeros((m, m))
        for k in range(25):
            ok = nb[k] >= 0
            np.add.at(A, (np.nonzero(ok)[0], nb[k][ok]), cf[k][ok])
        void = ~A.any(1)
        A[void, void] = 1.0
        ref = np.linalg.inv(A)
        got = inv[o:o + m * m].reshape(m, m)
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.cond(A) * np.linalg.norm(ref)
        assert np.array_equal(inv32[o:o + m * m].reshape(m, m), got.astype(np.float32))
        o += m * m
