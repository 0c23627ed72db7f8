"""What a context keeps between calls: the workspace over microstructures and numbers of right-hand
sides, against contexts that have seen one call only."""
import numpy as np
import pytest

import synth

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


def _equal_enriched_nodes(n=(60, 60, 80)):
    """Two level sets with the same number of enriched nodes and different numbers of cut tets: 1280
    isolated negative nodes (15 enriched nodes, 24 cut tets each) and a slab of negative planes (its four
    bounding node planes)."""
    few = np.ones(n)
    few.reshape(-1)[np.ravel_multi_index(
        [v.ravel()[:1280] for v in np.meshgrid(*[np.arange(0, m - 2, 3) for m in n], indexing="ij")], n)] = -0.7
    many = np.ones(n)
    many[20:40] = -0.7
    return n, few, many


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_more_cut_tets_on_the_same_enriched_nodes(xf, precision):
    """The partial sums grow with the cut tets while the vectors stay as long as they were.  Applies
    agree to rounding (1e-12, FP32 2e-5), stresses to ten times the solver's tolerance, gradients (of first
    order in the fields' error, in part FP32) to a few FP32 roundings."""
    n, few, many = _equal_enriched_nodes()
    kept, fresh = xf.Solver(n, precision=precision), xf.Solver(n, precision=precision)
    kept.set_microstructure(few, LM, LP)
    fresh.set_microstructure(many, LM, LP)
    rng = np.random.default_rng(3)
    d, eps = rng.normal(size=(8, kept.stride)), rng.normal(size=(8, 6))
    kept.apply(d, eps)
    kept.effective_stiffness()
    few_cut, nX = kept.num_cut_tets, kept.num_enriched
    kept.set_microstructure(many, LM, LP)
    assert kept.num_enriched == nX and kept.num_cut_tets > 1.5 * few_cut
    for prec, tol in (("fp64", 1e-12), ("fp32", 2e-5)):
        (q, sig), (q0, sig0) = (s.apply(d, eps, precision=prec) for s in (kept, fresh))
        assert _rel(q, q0) < tol and _rel(sig, sig0) < tol
    (a, b) = (s.solve(eps, u=False)["mean_stress"] for s in (kept, fresh))
    assert _rel(a, b) < 1e-9
    (C, st), (C0, st0) = (s.effective_stiffness() for s in (kept, fresh))
    assert st["converged"] and st0["converged"] and _rel(C, C0) < 1e-9
    G = rng.normal(size=(6, 6))
    for x, x0 in zip(kept.grad(G), fresh.grad(G)):
        assert _rel(x, x0) < 1e-6
    kept.close()
    fresh.close()


def test_stress_integrals_of_sixty_four_right_hand_sides(xf):
    """The reduced sums of an apply (seven per right-hand side) at the largest number of right-hand
    sides, against the same vectors in groups of eight; the solve that follows is that of a fresh context."""
    n = (12, 10, 8)
    L = synth.sphere_levelset(n, (0.5, 0.45, 0.55), 0.3)
    s, fresh = xf.Solver(n), xf.Solver(n)
    for v in (s, fresh):
        v.set_microstructure(L, LM, LP)
    rng = np.random.default_rng(5)
    d, eps = rng.normal(size=(64, s.stride)), rng.normal(size=(64, 6))
    q, sig = s.apply(d, eps)
    for r in range(0, 64, 8):
        q8, sig8 = fresh.apply(d[r:r + 8], eps[r:r + 8])
        assert _rel(q[r:r + 8], q8) < 1e-12 and _rel(sig[r:r + 8], sig8) < 1e-12
    (C, _), (C0, _) = s.effective_stiffness(), fresh.effective_stiffness()
    assert _rel(C, C0) < 1e-9
    s.close()
    fresh.close()


def test_captured_apply_outlives_the_reduced_records(xf):
    """An FP64 apply captured by the caller, replayed before and after a call whose buffers push the
    reduced cut-tet records out of the memory cap, over caps a quarter of the records apart: the replays
    agree with the eager apply (1e-12) and with each other, also once the freed memory holds NaN."""
    import torch
    n = (16, 12, 10)
    L = synth.sphere_levelset(n, (0.5, 0.45, 0.55), 0.3)
    ref = xf.Solver(n)
    ref.set_microstructure(L, LM, LP)
    ncut = ref.num_cut_tets
    big = np.random.default_rng(2).normal(size=(24, ref.stride))
    qb, sb = ref.apply(big)
    ref.close()
    d = torch.from_numpy(big[:2]).cuda()
    served = refused = 0
    for cap in range(4 << 20, 48 << 20, 256 * ncut):
        st = torch.cuda.Stream()
        s = xf.Solver(n, max_device_bytes=cap, stream=st)
        try:
            s.set_microstructure(L, LM, LP)
        except xf.XfftError as e:
            assert e.status == xf.capi.XFFT_ENOMEM
            s.close()
            continue
        q = torch.full_like(d, float("nan"))
        out = torch.full((2, 7), float("nan"), dtype=torch.float64, device="cuda")
        s.apply_noalloc(d, q, out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            s.apply_noalloc(d, q, out)
        for after in (False, True):
            if after:
                try:
                    assert _rel(s.apply(big)[0], qb) < 1e-12
                    served += 1
                except xf.XfftError as e:
                    assert e.status == xf.capi.XFFT_ENOMEM
                    refused += 1
                junk = [torch.full((1024 * ncut // 16,), float("nan"), dtype=torch.float64, device="cuda")
                        for _ in range(4)]
            q.fill_(float("nan"))
            out.fill_(float("nan"))
            graph.replay()
            torch.cuda.synchronize()
            assert _rel(q.cpu().numpy(), qb[:2]) < 1e-12, (cap, after)
            assert _rel(out.cpu().numpy()[:, 1:], sb[:2]) < 1e-12, (cap, after)
        del junk, graph
        s.close()
    assert served >= 4 and refused >= 1


def test_green_table_is_counted_and_gives_way(xf):
    """The line passes' Green table (9 reals per frequency) counts towards max_device_bytes and is only taken
    where it fits: a context whose cap is below its size holds next to nothing, and over caps from the smallest
    that a preconditioner call fits in, a quarter of the table apart, the results are those without
    a cap (1e-11 and 2e-5 of their norm for the other way of forming the inverses)."""
    import torch
    n = (90, 60, 50)
    table = 9 * n[0] * n[1] * (n[2] // 2 + 1)
    L = synth.sphere_levelset(n, (0.5, 0.45, 0.55), 0.3)
    for precision, size, tol in (("fp64", 8 * table, 1e-11), ("fp32", 4 * table, 2e-5)):
        s = xf.Solver(n, precision=precision)
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        capped = [xf.Solver(n, precision=precision, max_device_bytes=size - 1) for _ in range(4)]
        torch.cuda.synchronize()
        assert free0 - torch.cuda.mem_get_info()[0] < 4 * size - (2 << 20)
        for c in capped:
            c.close()
        s.set_microstructure(L, LM, LP)
        f = np.random.default_rng(4).normal(size=(2, s.stride))
        for c in range(3):
            f[:, c * s.N:(c + 1) * s.N] -= f[:, c * s.N:(c + 1) * s.N].mean(1, keepdims=True)
        ref, rr = s.precondition(f, precision=precision)
        C0 = s.effective_stiffness()[0]
        s.close()

        def serves(cap):
            s = xf.Solver(n, precision=precision, max_device_bytes=cap)
            try:
                s.set_microstructure(L, LM, LP)
                z, zr = s.precondition(f, precision=precision)
                assert _rel(z, ref) < tol and _rel(zr, rr) < 10 * tol
                return True
            except xf.XfftError as e:
                assert e.status == xf.capi.XFFT_ENOMEM
                return False
            finally:
                s.close()

        low, high = 0, 1 << 30
        while high - low > size // 4:
            mid = (low + high) // 2
            low, high = (low, mid) if serves(mid) else (mid, high)
        assert all(serves(high + k * (size // 4)) for k in range(7))
        s = xf.Solver(n, precision=precision, max_device_bytes=1 << 30)
        s.set_microstructure(L, LM, LP)
        assert _rel(s.effective_stiffness()[0], C0) < 1e-9
        s.close()


@pytest.mark.parametrize("n", [(16, 18, 20), (30, 12, 10), (150, 8, 6), (256, 6, 4)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_symbols_formed_in_the_pass(xf, n, precision):
    """A context has the Green table of its own precision; a preconditioner call in the other one forms the
    symbols in the pass.  Both against the oracle (1e-11 and 2e-5 of the norm) for each class of x lengths."""
    from oracle import XFEM
    ell = (1.0, 1.2, 0.9)
    L = np.ones(n)
    L[1, 2, 3] = -0.7
    s = xf.Solver(n, ell, precision=precision)
    s.set_microstructure(L, LM, LP)
    o = XFEM(L, n, ell, lame_minus=LM, lame_plus=LP)
    f = np.random.default_rng(6).normal(size=(2, s.stride))
    for c in range(3):
        f[:, c * s.N:(c + 1) * s.N] -= f[:, c * s.N:(c + 1) * s.N].mean(1, keepdims=True)
    for prec, tol in (("fp64", 1e-11), ("fp32", 2e-5)):
        z, _ = s.precondition(f, precision=prec)
        for k in range(2):
            assert _rel(z[k], o.precondition(f[k], green="fft")) < tol, prec
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_first_blocks_have_their_exact_size(xf, precision):
    """A context without a cap takes no more device memory for its first microstructure and solve than one
    with a cap that it stays below, and after a second, smaller microstructure no more than a third above
    (the driver hands out 2 MB pieces: 24 MB of tolerance for some fifty blocks of a gigabyte)."""
    import torch
    n = (96, 96, 96)
    big, small = (np.minimum(synth.sphere_levelset(n, (0.3, 0.3, 0.3), r), synth.sphere_levelset(n, (0.8, 0.8, 0.8), r))
                  for r in (0.2, 0.18))
    used = []
    for cap in (1 << 34, 0):
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        s = xf.Solver(n, precision=precision, max_device_bytes=cap, autotune=False, tol=1e-4)
        use = []
        for L in (big, small):
            s.set_microstructure(L, LM, LP)
            assert s.effective_stiffness()[1]["converged"]
            torch.cuda.synchronize()
            use.append(free0 - torch.cuda.mem_get_info()[0])
        used.append(use)
        s.close()
    (e1, e2), (r1, r2) = used
    assert r1 <= e1 + (24 << 20), used
    assert r2 <= e2 * 4 / 3 + (24 << 20), used
