"""The FP64 and double-word stencil (csrc/apply_tile.cuh), the FP32 one (csrc/apply_kernels.cuh) and the
reduced cut-tet records (csrc/apply_cut_el.cuh) on grids at the edges of their tile shapes, against the
oracle's assembled operator: the smallest grid (a tile is a whole periodic axis), rows longer than a
block, one and several planes per item, ragged last tiles, uniform and unequal voxel edges, one and
eight right-hand sides.  Tolerances as for the other apply parity tests (1e-12, 1e-11, 2e-5 of the
result's norm)."""
import numpy as np
import pytest

import synth
from oracle import XFEM

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "dw": 1e-11, "fp32": 2e-5}


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


def _problem(n, uniform):
    ell = tuple(v / max(n) for v in n) if uniform else (1.0, 1.3, 0.7)
    c = [0.45 * e for e in ell]
    L = synth.sphere_levelset(n, c, 0.31 * min(ell), ell)
    return ell, L, synth.lame_from_E_nu(20.0, 0.2), synth.lame_from_E_nu(1.0, 0.3), synth.voxel_scale(n, 5)


@pytest.mark.parametrize("n,uniform,k", [((4, 4, 4), True, 1), ((4, 6, 4), False, 8), ((6, 4, 160), True, 2),
                                         ((36, 6, 10), False, 1), ((18, 30, 36), True, 3), ((4, 144, 6), False, 2)])
def test_apply_at_tile_edges(xf, n, uniform, k):
    ell, L, lm, lp, sc = _problem(n, uniform)
    o = XFEM(L, n, ell, lame_minus=lm, lame_plus=lp, scale=sc)
    o.assemble()
    rng = np.random.default_rng(sum(n) + k)
    d = rng.normal(size=(k, o.ndof))
    eps = rng.normal(size=(k, 6))
    ref = (o.A @ d.T).T
    tot = ref + np.stack([o.rhs(e) for e in eps])
    sref = np.stack([np.asarray(o.Sm @ v).ravel() + o.Cbar @ e for v, e in zip(d, eps)])
    for solver in ("fp64", "fp32"):  # FP64 applies of a mixed-precision solver use the moment records
        s = xf.Solver(n, ell, precision=solver)
        s.set_microstructure(L, lm, lp, sc)
        for prec, tol in TOL.items():
            q, sig = s.apply(d, precision=prec)
            qt, sigt = s.apply(d, eps=eps, precision=prec)
            for r in range(k):
                assert _rel(q[r], ref[r]) < tol, (solver, prec)
                assert _rel(qt[r], tot[r]) < tol, (solver, prec)
                assert _rel(sigt[r], sref[r]) < tol, (solver, prec)
        s.close()


def test_double_word_split_of_small_values(xf):
    """Values below 2^-73 leave the integer split of doubles; zeros and large ones stay in it."""
    n = (8, 6, 10)
    ell, L, lm, lp, sc = _problem(n, False)
    o = XFEM(L, n, ell, lame_minus=lm, lame_plus=lp, scale=sc)
    o.assemble()
    d = np.random.default_rng(2).normal(size=(3, o.ndof)) * np.array([[1e-24], [1.0], [1e12]])
    d[1, ::3] = 0.0
    s = xf.Solver(n, ell)
    s.set_microstructure(L, lm, lp, sc)
    q, _ = s.apply(d, precision="dw")
    for r in range(3):
        assert _rel(q[r], o.A @ d[r]) < 1e-11


def test_reduced_records_give_way_to_a_memory_cap(xf):
    """Down to the smallest cap that a solve fits in, the solution is that without a cap: where the
    reduced records do not fit beside the workspace the moment records serve."""
    n = (16, 12, 10)
    ell, L, lm, lp, sc = _problem(n, False)
    s = xf.Solver(n, ell)
    s.set_microstructure(L, lm, lp, sc)
    ref, ncut = s.effective_stiffness()[0], s.num_cut_tets
    s.close()
    cap, fits, low = 16 << 20, 0, None
    while low is None:
        s = xf.Solver(n, ell, max_device_bytes=cap)
        try:
            s.set_microstructure(L, lm, lp, sc)
            C, st = s.effective_stiffness()
            assert st["converged"] and _rel(C, ref) < 1e-9
            fits += 1
        except xf.XfftError as e:
            assert e.status == xf.capi.XFFT_ENOMEM
            low = cap
        s.close()
        cap -= 256 * ncut  # a quarter of the reduced records
    assert fits >= 4
