"""Inner products and norms per right-hand side (csrc/blas.cu: dot_partial_k, blocks by the length) at lengths of
one block, a part of one, several with a remainder, and more than the most blocks take.

The FP32 forms, which no public call reaches alone, run in a small program linked against the library.

Tolerance: a thread's sum of at most some 100 products and the tree above it, 128 x 2^-53 times the sum of the
products' magnitudes.  FP32: a product's own two roundings, 2 x 2^-24 of its magnitude at most; the sums keep
what they round off, so the bound does not grow with the terms.
"""
import subprocess

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, nrhs", [((2, 2, 2, 2), 3), ((5, 3, 4, 7), 2), ((8, 8, 8, 8), 5), ((7, 9, 11, 13), 1),
                                        ((24, 24, 24, 16), 1)])
@pytest.mark.parametrize("per_timeslice", [False, True])
def test_inner(dims, nrhs, per_timeslice):
    import torch

    import paper_1111_6288_gb300 as P

    a, b = (synth.gaussian_spinor(dims, nrhs, seed) for seed in (61, 62))
    ctx = P.Context(P.Params(dims=dims, m0=-1.5, eps=0.02, poly_degree=2, max_nrhs=nrhs))
    ctx.set_gauge(torch.from_numpy(synth.random_su3_field(dims, 0.3, seed=63)).cuda())
    got = P.inner(ctx, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), per_timeslice=per_timeslice)
    ctx.close()
    axes = tuple(range(2 if per_timeslice else 1, a.ndim))
    want = (a.conj() * b).sum(axis=axes)
    size = (np.abs(a) * np.abs(b)).sum(axis=axes)
    assert got.shape == want.shape
    assert np.all(np.abs(got - want) <= 128 * 2.0**-53 * size)


PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "ovl_internal.h"
int main(int argc, char** argv) {
    const long long n = atoll(argv[1]);
    const int nrhs = atoi(argv[2]);
    std::vector<float2> a(n * nrhs), b(n * nrhs);
    for (auto* p : {&a, &b}) {
        FILE* f = fopen(argv[p == &a ? 3 : 4], "rb");
        if (!f || fread(p->data(), sizeof(float2), p->size(), f) != p->size()) return 2;
        fclose(f);
    }
    float2 *da, *db;
    double2 *part, *out;
    cudaMalloc(&da, sizeof(float2) * a.size());
    cudaMalloc(&db, sizeof(float2) * b.size());
    cudaMalloc(&part, sizeof(double2) * ovl::kRedBlocks * nrhs);
    cudaMalloc(&out, sizeof(double2) * nrhs);
    cudaMemcpy(da, a.data(), sizeof(float2) * a.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(db, b.data(), sizeof(float2) * b.size(), cudaMemcpyHostToDevice);
    std::vector<double2> d(nrhs);
    std::vector<double> q(nrhs);
    ovl::dot_rhs<float>(da, db, n, nrhs, d.data(), part, out, 0);
    ovl::norm2_rhs<float>(da, n, nrhs, q.data(), part, out, 0);
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    for (int r = 0; r < nrhs; ++r) printf("%.17g %.17g %.17g\n", d[r].x, d[r].y, q[r]);
}
"""


@pytest.fixture(scope="module")
def run32(cuda_program, tmp_path_factory):
    exe, where = cuda_program(PROGRAM), tmp_path_factory.mktemp("dots")

    def run(a, b):
        for name, v in (("a", a), ("b", b)):
            v.astype(np.complex64).tofile(where / name)
        text = subprocess.run([str(exe), str(a.shape[1]), str(a.shape[0]), str(where / "a"), str(where / "b")], check=True,
                              capture_output=True, text=True).stdout
        v = np.array([[float(t) for t in line.split()] for line in text.splitlines()])
        return v[:, 0] + 1j * v[:, 1], v[:, 2]

    return run


# part of a block's 2048 elements, one block, a remainder, several, and more than 608 blocks of them
@pytest.mark.parametrize("n, nrhs", [(1, 2), (100, 3), (2047, 1), (2048, 2), (2049, 2), (98304, 2), (1300000, 1)])
def test_fp32_sums(run32, n, nrhs):
    rng = np.random.default_rng(n)
    a, b = ((rng.standard_normal((nrhs, n)) + 1j * rng.standard_normal((nrhs, n))).astype(np.complex64) for _ in "ab")
    a *= (2.0 ** rng.integers(-12, 13, (nrhs, n))).astype(np.float32)
    dot, norm = run32(a, b)
    a, b = a.astype(np.complex128), b.astype(np.complex128)
    size = (np.abs(a) * np.abs(b)).sum(axis=1)
    assert np.all(np.abs(dot - (a.conj() * b).sum(axis=1)) <= 2 * np.sqrt(2) * 2.0**-24 * size)
    want = (np.abs(a) ** 2).sum(axis=1)
    assert np.all(np.abs(norm - want) <= 2 * 2.0**-24 * want)


def test_fp32_sums_out_of_range(run32):
    """Products near the largest FP32 number, whose sums leave its range; one product that does; a NaN."""
    n = 98304
    a = np.full((4, n), 1.2e19, np.complex64)
    a[1] *= -1
    a[2, 77] = 3e19
    a[3, 99] = np.nan
    b = a.copy()
    b[1] *= -1
    dot, norm = run32(a, b)
    exact = n * np.float64(np.float32(1.2e19)) ** 2
    for got, want in ((norm[0], exact), (dot[0].real, exact), (dot[1].real, -exact), (norm[1], exact)):
        assert abs(got - want) <= 2 * 2.0**-24 * exact
    assert np.isposinf(norm[2]) and np.isposinf(dot[2].real) and dot[2].imag == 0.0
    assert np.isnan(norm[3]) and np.isnan(dot[3].real)
