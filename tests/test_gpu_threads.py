"""Several contexts at a time: grids whose line passes want different amounts of shared memory (above 48 KB:
200 x 60 x 96 and 144 x 60 x 108 in both precisions), in two host threads and in one batch, against
each alone.  Results of the same call agree to rounding (1e-11, FP32 2e-5 for the preconditioner; ten times
the solver's tolerance for stiffnesses)."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

GRIDS = [(200, 60, 96), (144, 60, 108)]


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


def _solver(xf, n, precision):
    ell = tuple(v / 100.0 for v in n)
    s = xf.Solver(n, ell, precision=precision)
    s.set_microstructure(synth.sphere_levelset(n, tuple(0.47 * v for v in ell), 0.4 * min(ell), ell),
                         synth.lame_from_E_nu(5.0, 0.25), synth.lame_from_E_nu(1.0, 0.3))
    return s


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_two_threads_precondition(xf, precision):
    solvers = [_solver(xf, n, precision) for n in GRIDS]
    rng = np.random.default_rng(1)
    f = []
    for s in solvers:
        v = rng.normal(size=(2, s.stride))
        for c in range(3):
            v[:, c * s.N:(c + 1) * s.N] -= v[:, c * s.N:(c + 1) * s.N].mean(1, keepdims=True)
        f.append(v)
    ref = [s.precondition(v, precision=precision)[0] for s, v in zip(solvers, f)]
    errors, gate = [], threading.Barrier(2)

    def work(k):
        try:
            gate.wait()
            for _ in range(20):
                z, _ = solvers[k].precondition(f[k], precision=precision)
                assert _rel(z, ref[k]) < (1e-11 if precision == "fp64" else 2e-5)
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for s in solvers:
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batch_of_two_line_grids(xf, precision):
    alone = []
    for n in GRIDS:
        s = _solver(xf, n, precision)
        alone.append(s.effective_stiffness()[0])
        s.close()
    solvers = [_solver(xf, n, precision) for n in GRIDS]
    C, st = xf.batch_effective_stiffness(solvers)
    for k in range(2):
        assert _rel(C[k], alone[k]) < 1e-9
    for s in solvers:
        s.close()
