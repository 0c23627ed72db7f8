"""Sums over voxels at the edges of the kernels that form them."""
import numpy as np
import pytest

import synth
from oracle import XFEM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2601_02172_gb300 as pkg
    return pkg


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


LM, LP = synth.lame_from_E_nu(10.0, 0.25), synth.lame_from_E_nu(1.0, 0.3)


@pytest.mark.parametrize("n", [(6, 6, 6), (10, 6, 6), (10, 10, 6), (8, 8, 4)])
def test_voxel_stress_of_a_partly_filled_warp(xf, n):
    """Numbers of voxels that leave 24, 8, 24 and 0 lanes of the last warp, each with one-phase and with
    cut voxels, against the oracle's stress of the same displacements (linear in them: rounding only)."""
    L = synth.sphere_levelset(n, (0.45, 0.5, 0.55), 0.3)
    s = xf.Solver(n)
    s.set_microstructure(L, LM, LP)
    o = XFEM(L, n, lame_minus=LM, lame_plus=LP)
    eps = np.random.default_rng(1).normal(size=(2, 6))
    out = s.solve(eps, voxel_stress=True)
    for r in range(2):
        u = np.concatenate([out["u_std"][r].ravel(), (out["u_enr"][r] / o.Dinvsqrt.T).ravel()])
        assert _rel(out["voxel_stress"][r], o.voxel_stress(u, eps[r]).T) < 1e-12
    s.close()


@pytest.mark.parametrize("n", [(18, 30, 36), (4, 6, 4), (6, 4, 160)])
@pytest.mark.parametrize("mean", [0.0, 1e6, 1e9])
def test_energy_of_displacements_with_a_mean(xf, n, mean):
    """<d, A d> of the allocation-free apply for smooth and for random d on a large constant, against the
    oracle's operator on d without it (subtracted exactly: d is a multiple of the constant's last place).
    Differences of neighbours are exact there, so the result is good to the rounding of its sums (1e-12)."""
    import torch
    ell = tuple(v / max(n) for v in n)
    L = synth.sphere_levelset(n, tuple(0.45 * e for e in ell), 0.31 * min(ell), ell)
    s = xf.Solver(n, ell)
    s.set_microstructure(L, LM, LP)
    o = XFEM(L, n, ell, lame_minus=LM, lame_plus=LP)
    o.assemble()
    x = np.stack(np.meshgrid(*[np.arange(m) / m for m in n], indexing="ij"))
    rng = np.random.default_rng(7)
    d = rng.normal(size=(2, s.stride))
    for c in range(3):
        d[0, c * s.N:(c + 1) * s.N] = (np.sin(2 * np.pi * x[c]) + np.cos(2 * np.pi * x[c - 1])).ravel()
        d[:, c * s.N:(c + 1) * s.N] += mean * (1 + c)
    e = d.copy()
    for c in range(3):
        e[:, c * s.N:(c + 1) * s.N] -= mean * (1 + c)
    out = torch.empty((2, 7), dtype=torch.float64, device="cuda")
    dd = torch.from_numpy(d).cuda()
    s.apply_noalloc(dd, torch.empty_like(dd), out)
    for k in range(2):
        ref = float(e[k] @ (o.A @ e[k]))
        assert abs(float(out[k, 0]) - ref) < 1e-12 * ref, k
    s.close()
