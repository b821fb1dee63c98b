"""Bounded waits of the single-precision march (csrc/hz_march.cuh) that run out.

HZ_COPY_TEST=1 at handle creation makes every wait for a plane's copy expect an
arrival that never comes, with a short poll limit.  The copies themselves are the
ordinary ones and land; the kernel has to stop copying, let what it asked for
land, and end.
"""
import pytest

import hz_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def hz():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    return hz


def _solver(hz, n, nrhs, monkeypatch, give_up):
    w = W.gaussian_lens(n=n, n_pml=8)
    if give_up:
        monkeypatch.setenv("HZ_COPY_TEST", "1")
    s = hz.Solver(w.n, w.n_pml, w.h, w.omega, w.c, params=hz.default_params(autotune=0, max_pc=2, max_refine=1),
                  max_nrhs=nrhs)
    monkeypatch.delenv("HZ_COPY_TEST", raising=False)
    return w, s


@pytest.mark.parametrize("nrhs", [1, 2])
def test_march_waits_give_up_and_are_reported(hz, monkeypatch, nrhs):
    """105^3: apply, residual and (two right-hand sides) Jacobi map are marches.
    Every call returns, the context stays usable, a solve on the handle reports
    HZ_ETIMEOUT, and another handle's results are right."""
    w, s = _solver(hz, 104, nrhs, monkeypatch, True)
    x = torch.from_numpy(W.random_complex((nrhs,) + s.level_shape[0], 3)).to("cuda", torch.complex64)
    s.iofd_apply(x)
    s.iofd_apply(x, op=hz.HZ_OP_B)
    s.residual_static(x, x.clone())
    s.iofd_jacobi(x)
    torch.cuda.synchronize()
    with pytest.raises(hz.HzError) as e:
        s.helmholtz_solve(w.sources * nrhs)
    assert e.value.status == hz.HZ_ETIMEOUT, e.value
    s.close()
    _, t = _solver(hz, 104, nrhs, monkeypatch, False)
    y, ref = t.iofd_apply(x), t.iofd_apply(x.to(torch.complex128))
    assert float(torch.linalg.vector_norm(y.to(torch.complex128) - ref) / torch.linalg.vector_norm(ref)) <= 2e-6
    t.close()


def test_earlier_give_up_is_not_reported_by_a_correct_solve(hz, monkeypatch):
    """49^3: the window apply is a march whose waits run out, a solve runs no march.
    The solve is right and returns so; hz_check reports the window apply, once."""
    w = W.gaussian_lens(n=48, n_pml=8)
    monkeypatch.setenv("HZ_COPY_TEST", "1")
    s = hz.Solver(w.n, w.n_pml, w.h, w.omega, w.c, params=hz.default_params(tol=1e-6))
    monkeypatch.delenv("HZ_COPY_TEST")
    x = torch.zeros((1, 51) + s.level_shape[0][1:], dtype=torch.complex64, device="cuda")
    s.check()
    for check_first in (True, False):
        s.iofd_apply_window(x, 0, 49)
        if check_first:
            with pytest.raises(hz.HzError) as e:
                s.check()
            assert e.value.status == hz.HZ_ETIMEOUT
        _, _, st = s.helmholtz_solve(w.sources, want_u=False)
        assert st["rel_res"] <= 1e-6
        if not check_first:
            with pytest.raises(hz.HzError) as e:
                s.check()
            assert e.value.status == hz.HZ_ETIMEOUT
        s.check()
    s.close()
