"""The preconditioner's line passes (csrc/fft_lines.cuh) on lengths at the edges of their plans,
against the oracle's FFT preconditioner on random mean-free fields: one, two and three factors on
each axis, odd half lengths along z, the smallest and largest lengths, tiles that do not divide the
columns, and an odd number of enriched DOFs (right-hand sides on odd offsets).  Tolerances as for the
other preconditioner parity tests: 1e-11 (FP64) and 2e-5 (FP32) of the result's norm."""
import numpy as np
import pytest

import synth
from oracle import XFEM

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 4), (6, 10, 4), (54, 50, 60), (18, 16, 90), (36, 250, 20), (30, 480, 6), (486, 6, 10),
          (6, 6, 750), (640, 4, 6), (1024, 4, 4), (4, 1024, 4), (4, 4, 1024)]


@pytest.fixture(scope="module")
def xf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2601_02172_gb300 as pkg
    return pkg


@pytest.mark.parametrize("n", SHAPES)
def test_line_passes_match_the_oracle(xf, n):
    ell = (1.0, 1.2, 0.9)
    L = np.ones(n)
    L[1, 2, 3] = -0.7  # one negative node: 15 enriched nodes, an odd stride
    lm, lp = synth.lame_from_E_nu(5.0, 0.3), synth.lame_from_E_nu(1.0, 0.3)
    s = xf.Solver(n, ell)
    s.set_microstructure(L, lm, lp)
    assert s.num_enriched % 2 == 1
    o = XFEM(L, n, ell, lame_minus=lm, lame_plus=lp)
    N = n[0] * n[1] * n[2]
    f = np.random.default_rng(N + n[0]).normal(size=(3, s.stride))
    for c in range(3):
        f[:, c * N:(c + 1) * N] -= f[:, c * N:(c + 1) * N].mean(1, keepdims=True)
    ref = np.stack([o.precondition(v, green="fft") for v in f])
    for prec, tol in (("fp64", 1e-11), ("fp32", 2e-5)):
        z, rr = s.precondition(f, precision=prec)
        for k in range(3):
            assert np.linalg.norm(z[k] - ref[k]) < tol * np.linalg.norm(ref[k]), (prec, k)
            assert abs(rr[k] - f[k] @ ref[k]) < 10 * tol * abs(f[k] @ ref[k]), (prec, k)
