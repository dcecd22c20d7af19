"""FP64 calls on a device without the memory that fixed point takes beyond FP64 (links of 576 B a site, of 144 B a
site and field phase, vectors of 196 instead of 192 B a site and one more of them): the recurrence runs in FP64 instead,
to the same results.  The device's answer is faked on the host: a preloaded cudaMalloc refuses given sizes.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
int cudaMalloc(void** p, size_t n) {
    static int (*real)(void**, size_t);
    const char* refused = getenv("REFUSED_SIZES");
    char size[32];
    snprintf(size, sizeof(size), ",%zu,", n);
    if (refused && strstr(refused, size)) {
        fprintf(stderr, "refused %zu\n", n);
        return 2; /* cudaErrorMemoryAllocation */
    }
    if (!real) real = (int (*)(void**, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
    return real(p, n);
}
"""

PROGRAM = r"""
import sys
import numpy as np
import torch
import synth
import paper_1111_6288_gb300 as P
dims = (4, 4, 4, 6)
ctx = P.Context(P.Params(dims=dims, bc=(0, 0, 0, 1), m0=-1.5, eps=0.1, poly_degree=8, max_nrhs=4))
ctx.set_gauge(torch.from_numpy(synth.random_su3_field(dims, 0.3, seed=81)).cuda())
P.deflate(ctx, None, [], phase=0.2)
out = {}
for nrhs in (3, 1, 3):
    x = torch.from_numpy(synth.gaussian_spinor(dims, nrhs, 82)).cuda()
    for name, f in (("sign", lambda v, y: P.apply_sign_Hw(ctx, v, y, phase=[0.2] * nrhs)),
                    ("derivative", lambda v, y: P.apply_dDdphi(ctx, v, y, 0.1, phase=[0.2] * nrhs))):
        y = torch.empty_like(x)
        f(x, y)
        out[f"{name}{nrhs}"] = y.cpu().numpy()
out["eigenvalues"] = np.asarray(P.eigensolve_Q(ctx, 2, tol=1e-9)[0])
np.savez(sys.argv[1], **out)
"""


def test_refused_memory(tmp_path):
    from paper_1111_6288_gb300 import build

    V = 4 * 4 * 4 * 6
    tiles = V // 32
    vector, links = (12 * 16 + 4) * 32 * tiles, 4 * 9 * 16 * 32 * tiles + 64
    (tmp_path / "shim.c").write_text(SHIM)
    (tmp_path / "run.py").write_text(PROGRAM)
    shim = tmp_path / "shim.so"
    subprocess.run(["gcc", "-shared", "-fPIC", str(tmp_path / "shim.c"), "-o", str(shim), "-ldl"], check=True)

    def run(name, sizes):
        env = dict(os.environ, LD_PRELOAD=str(shim), PYTHONPATH=build.ROOT,
                   REFUSED_SIZES="," + "".join(f"{n}," for n in sizes))
        r = subprocess.run([sys.executable, str(tmp_path / "run.py"), str(tmp_path / name)], env=env, capture_output=True,
                           text=True, cwd=build.ROOT)
        assert r.returncode == 0, r.stderr
        assert ("refused" in r.stderr) == bool(sizes)
        return dict(np.load(tmp_path / (name + ".npz")))

    want = run("all", [])
    for name, sizes in (("links", [links]), ("field", [(links - 64) // 4]), ("three", [3 * vector]),
                        ("every", [vector * k for k in range(1, 40)])):
        got = run(name, sizes)
        for key in want:
            # both routes to FP64's accuracy: 8 (2 n + 1) (n + 1) 2^-53, the derivative's terms grow by n + 1 once more
            tol = 8 * 17 * 9 * 9 * 2.0**-53 if "value" not in key else 1e-9
            assert np.linalg.norm(got[key] - want[key]) <= tol * np.linalg.norm(want[key]), (name, key)
