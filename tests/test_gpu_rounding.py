"""Rounding of the complex64 operators.

Fine level: both kernel families (gather form at 49^3, march at 85^3 and 105^3)
against the complex128 kernels.  u = 2^-24 = 6e-8.  A row's centre term carries the
rounding of a tabulated weight and of its evaluation (u / sqrt(3) each in the root
mean square), the sum one of its own when the far shells are added first; the centre
is up to 1.3 times the row on a random field.  sqrt(3) * u / sqrt(3) * 1.3 = 8e-8.
Weights formed per row from several rounded tables, or the centre added first, exceed
it.

Adjoint on the 4h level, where kappa^2 M dominates: the rounding of the local
coordinate counts twice, then weight, evaluation, product and sum: sqrt(4 + 4) *
u / sqrt(3), and the centre is up to 1.5 times the row: 1.5e-7.  A coordinate off by
the rounding of 1 / 2 pi (4e-8, twice) exceeds it.
"""
import math

import pytest

import hz_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -24
ROW, ADJ4 = 1.3 * U, 1.5 * U * math.sqrt(8.0 / 3.0)


def _rel(a, b):
    return float(torch.linalg.vector_norm(a.to(torch.complex128) - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("n,pml,nrhs", [(48, 8, 1), (84, 8, 1), (104, 8, 2)])
@pytest.mark.parametrize("homogeneous", [True, False])
def test_fine_level_rounding(n, pml, nrhs, homogeneous):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    gen = torch.Generator("cuda").manual_seed(11)
    c = torch.rand((n + 1,) * 3, dtype=torch.float64, device="cuda", generator=gen)
    c = 1.5 + (0.0 if homogeneous else 1.0) * c
    h, omega = W.grid_params(n, pml, 1.5)
    s = hz.Solver(n, pml, h, omega, c, params=hz.default_params(autotune=0), max_nrhs=nrhs)
    x = torch.randn((nrhs,) + s.level_shape[0], dtype=torch.complex64, device="cuda", generator=gen)
    g = torch.randn(x.shape, dtype=torch.complex64, device="cuda", generator=gen)
    x128, g128 = x.to(torch.complex128), g.to(torch.complex128)
    err = {}
    for name, op in (("A", hz.HZ_OP_A), ("B", hz.HZ_OP_B)):
        err["apply " + name] = _rel(s.iofd_apply(x, op=op), s.iofd_apply(x128, op=op)) / ROW
        err["residual " + name] = _rel(s.residual_static(g, x, op=op)[0], s.residual_static(g128, x128, op=op)[0]) / ROW
    s.close()
    assert max(err.values()) <= 1.0, err


def test_adjoint_rounding_on_the_4h_level():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    gen = torch.Generator("cuda").manual_seed(12)
    c = 1.5 + torch.rand((145,) * 3, dtype=torch.float64, device="cuda", generator=gen)
    h, omega = W.grid_params(144, 8, 1.5)
    s = hz.Solver(144, 8, h, omega, c, params=hz.default_params(autotune=0))
    x = torch.randn((1,) + s.level_shape[2], dtype=torch.complex64, device="cuda", generator=gen)
    for op in (hz.HZ_OP_A_ADJ, hz.HZ_OP_B_ADJ):
        err = _rel(s.iofd_apply(x, op=op, level=2), s.iofd_apply(x.to(torch.complex128), op=op, level=2))
        assert err <= ADJ4, (op, err)
    s.close()
