"""The Wilson kernel that stages whole x-rows in shared memory (bulk copies on an mbarrier).

On lattices whose x-rows tile a thread block (Lx a multiple of 4, rows x Lx a multiple of 32
sites), launch_shape | 32 selects it.  It must agree with the oracle like the plain kernel and
give the same bits as the plain kernel, which accumulates the hops in the same order (z, t,
x, y), for every right-hand-side block and register budget, in FP32 and 16-bit storage.
"""
from __future__ import annotations

import subprocess

import numpy as np
import pytest

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu

M0 = -1.5
BC_NUM = {0: 1.0, 1: -1.0, 2: 0.0}
DIMS, BC = (8, 8, 4, 6), (2, 0, 1, 2)  # 384-site slices of 8 rows; Dirichlet x, t, antiperiodic z
PHASES = [0.3, 0.0, -0.2]
TOL = {1: 2e-6, 2: 16 * 2.0 ** -11, 3: 16 * 2.0 ** -8}  # one H_w (see test_gpu_parity / test_gpu_half)
TILED = [1 | 32, 1 | 16 | 32, 2 | 32, 4 | 32]


def obc(bc):
    return tuple(BC_NUM[b] for b in bc)


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1111_6288_gb300 as P

    return P


def ctx_for(P, precision, shape, degree=16, eps=0.05):
    import torch

    ctx = P.Context(P.Params(dims=DIMS, bc=BC, m0=M0, eps=eps, poly_degree=degree, precision=precision,
                             inner_precision=1, max_nrhs=4, launch_shape=shape))
    ctx.set_gauge(torch.from_numpy(synth.random_su3_field(DIMS, 0.3, 31)).cuda())
    for ph in set(PHASES):
        P.deflate(ctx, None, [], phase=ph)  # empty small spaces: the polynomial acts on everything
    return ctx


def run(P, ctx, fn, x, **kw):
    import torch

    xd = torch.from_numpy(np.ascontiguousarray(x)).to(torch.complex64).cuda()
    out = torch.empty_like(xd)
    fn(ctx, xd, out, **kw)
    P.sync(ctx)
    return out.cpu().numpy()


# One H_w on the launch shape given (single applications through the library's calls take no tiles).
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <type_traits>
#include <vector>
#include "ovl_internal.h"
using namespace ovl;
template <typename T>
T* upload(const char* path, size_t n) {
    std::vector<T> h(n);
    FILE* f = fopen(path, "rb");
    if (!f || fread(h.data(), sizeof(T), n, f) != n) exit(2);
    fclose(f);
    T* d;
    cudaMalloc(&d, n * sizeof(T));
    cudaMemcpy(d, h.data(), n * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}
void* device(size_t bytes) {
    void* d = nullptr;
    if (cudaMalloc(&d, bytes) != cudaSuccess) exit(3);
    return d;
}
template <typename S>
void apply(const Geom& g, double m0, const void* U, const void* x, const double* phase, int nrhs, int shape, void* y) {
    const size_t n = 96ull * g.V * nrhs;  // bytes in FP32
    void *links = device(192ull * g.V), *in = device(n), *out = device(n), *y32 = device(n);
    if constexpr (std::is_same<S, float>::value) launch_pack_gauge<float>(U, 0, links, g, 0);
    else launch_pack_gauge_half<S>(U, 0, links, g.V, 0);
    launch_pack_spinor<S>(x, 1, in, g.V, nrhs, 0);
    launch_dslash<S>(g, m0, links, in, out, nrhs, phase, Epilogue(), 0, false, shape);
    if constexpr (std::is_same<S, float>::value) y32 = out;
    else launch_from_half<S>(out, y32, g.V, nrhs, 0);
    launch_unpack_spinor<float>(y32, y, 1, g.V, nrhs, 0);
}
int main(int, char** v) {  // precision shape nrhs L[4] bcf[4] m0 U x phase y
    Geom g;
    g.V = 1;
    for (int k = 0; k < 4; ++k) g.V *= g.L[k] = atoi(v[4 + k]), g.bcf[k] = atof(v[8 + k]);
    const int precision = atoi(v[1]), shape = atoi(v[2]), nrhs = atoi(v[3]);
    const double m0 = atof(v[12]);
    const double2* U = upload<double2>(v[13], 36ull * g.V);
    const float2* x = upload<float2>(v[14], 12ull * g.V * nrhs);
    const double* phase = upload<double>(v[15], nrhs);
    std::vector<float2> y(12ull * g.V * nrhs);
    void* dy = device(y.size() * sizeof(float2));
    if (precision == 1) apply<float>(g, m0, U, x, phase, nrhs, shape, dy);
    else if (precision == 2) apply<H16>(g, m0, U, x, phase, nrhs, shape, dy);
    else apply<B16>(g, m0, U, x, phase, nrhs, shape, dy);
    if (cudaMemcpy(y.data(), dy, y.size() * sizeof(float2), cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
    FILE* f = fopen(v[16], "wb");
    fwrite(y.data(), sizeof(float2), y.size(), f);
    fclose(f);
    printf("%d %d\n", tile_rows(g, shape & kShapeRhsMask), take_wait_timeouts());
}
"""


@pytest.fixture(scope="module")
def one_application(cuda_program, tmp_path_factory):
    exe, where = cuda_program(PROGRAM), tmp_path_factory.mktemp("tiled")

    def run_one(precision, shape, U, x):
        U.astype(np.complex128).tofile(where / "U")
        x.astype(np.complex64).tofile(where / "x")
        np.array(PHASES[:len(x)]).tofile(where / "phase")
        args = [precision, shape, len(x), *DIMS, *obc(BC), M0] + [where / k for k in ("U", "x", "phase", "y")]
        rows, timeouts = (int(t) for t in subprocess.run([str(a) for a in [exe] + args], check=True, capture_output=True,
                                                         text=True).stdout.split())
        assert timeouts == 0
        return np.fromfile(where / "y", np.complex64).reshape(x.shape), rows

    return run_one


@pytest.mark.parametrize("precision", [1, 2, 3])
@pytest.mark.parametrize("shape", TILED)
def test_tiled_wilson_matches_oracle(P, one_application, precision, shape):
    U = synth.random_su3_field(DIMS, 0.3, 31)
    x = synth.gaussian_spinor(DIMS, 3, 32)
    got, rows = one_application(precision, shape, U, x)
    assert rows > 0  # the lattice allows the tiled kernel for this shape
    want = np.stack([dirac.hermitian_wilson(U, x[j], M0, obc(BC), PHASES[j]) for j in range(3)])
    err = float(np.abs(got - want).max() / np.abs(want).max())
    assert err < TOL[precision], err
    plain, _ = one_application(precision, shape & 15, U, x)
    assert np.array_equal(plain, got)


@pytest.mark.parametrize("precision", [1, 2, 3])
def test_tiled_overlap_equals_plain_bitwise(P, precision):
    """D(m) through the whole recurrence: the plain one-system kernel, every tiled shape on the
    batch of three, and one system at a time with the tiled kernel give the same bits."""
    x = synth.gaussian_spinor(DIMS, 3, 33)
    ref = run(P, ctx_for(P, precision, 1), P.apply_overlap, x, mass=0.05, phase=PHASES)
    assert np.isfinite(ref).all() and np.abs(ref).max() > 0
    for shape in TILED:
        ctx = ctx_for(P, precision, shape)
        assert np.array_equal(run(P, ctx, P.apply_overlap, x, mass=0.05, phase=PHASES), ref), shape
        one = run(P, ctx, P.apply_overlap, x[1:2], mass=0.05, phase=PHASES[1:2])
        assert np.array_equal(one[0], ref[1]), shape
        ctx.close()


def test_tuner_offers_the_tiled_kernel(P):
    import torch

    ctx = ctx_for(P, 1, 0)
    x = torch.from_numpy(synth.gaussian_spinor(DIMS, 2, 34)).to(torch.complex64).cuda()
    P.apply_sign_Hw(ctx, x, torch.empty_like(x), phase=[0.0, 0.0])
    P.sync(ctx)
    assert "t:" in ctx.tune_info
    ctx.close()
