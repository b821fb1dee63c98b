"""The single-sweep Jacobi kernel of the march, A on the fine and B on the 2h level,
one and two right-hand sides per block.

165^3: the 2h level has 83^3 nodes.  Three sweeps on every level are one two-sweep map
and one single sweep.  One Krylov step per level: some 30 stencil passes in a row, each
within 1.2e-7 of its complex128 value, and small least-squares solves that amplify by no
more than a few: 30 * 1.2e-7 * 3 = 1.1e-5.
"""
import pytest

import hz_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [2, 3])
def test_three_sweeps_march_on_two_levels(nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    p = hz.default_params(autotune=0, nJ_h=3, nJ_2h=3, nJ_4h=3, m_h=1, c_2h=1, m_2h=1, m_4h=1)
    gen = torch.Generator("cuda").manual_seed(8)
    c = 1.5 + torch.rand((165,) * 3, dtype=torch.float64, device="cuda", generator=gen)
    h, omega = W.grid_params(164, 8, 1.5)
    s = hz.Solver(164, 8, h, omega, c, params=p, max_nrhs=nrhs)
    r = torch.randn((nrhs,) + s.level_shape[0], dtype=torch.complex64, device="cuda", generator=gen)
    z, ref = s.threegrid_precond(r), s.threegrid_precond(r.to(torch.complex128))
    assert float(torch.linalg.vector_norm(z.to(torch.complex128) - ref) / torch.linalg.vector_norm(ref)) <= 1.1e-5
    s.close()
