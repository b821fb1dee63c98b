"""Tile edges of the adjoint and small-grid kernels, and coarse weight tables.

Grids on both sides of the 2^17 nodes below which the forward and adjoint
kernels take 8 x 8 tiles, with ragged and exact last tiles, PML layers narrower
and wider than a tile, none at all, and two and three right-hand sides.

Tolerances (u the unit roundoff): a row sums 27 products whose weights are a few
roundings from exact, at most about 40 u sum |w||x|, and sum |w||x| is two to
three times |row| in the root mean square: 120 u.  complex128 (u = 1.1e-16)
keeps the adjoint identity to 1.4e-14 of ||A x|| ||y||, and the two sides add up
to twice that: 3e-14.  complex64 (u = 6e-8): 2e-6 is below that worst case.
"""
import numpy as np
import pytest

import hz_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL128, TOL64 = 3e-14, 2e-6


def _solver(shape, pml, nrhs, **kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    nx, ny, nz = shape
    c = 1.5 + np.random.default_rng(5).random((nz + 1, ny + 1, nx + 1))
    h, omega = W.grid_params(min(shape), pml, 1.5)
    return hz, hz.Solver(shape, pml, h, omega, c, params=hz.default_params(autotune=0), max_nrhs=nrhs, **kw)


def _rel(a, b):
    return float(torch.linalg.vector_norm(a.to(torch.complex128) - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("shape,pml,nrhs", [
    ((24, 24, 24), 4, 1),       # 25 = 3 * 8 + 1 columns, levels of 13 and 7
    ((28, 60, 12), 4, 2),       # 29 x 61 x 13
    ((52, 52, 44), 12, 3),      # 126405 nodes: the last small ones; PML wider than a tile
    ((52, 52, 48), 4, 1),       # 137641 nodes: 32 x 8 tiles
    ((64, 60, 92), 0, 2),       # 65 = 2 * 32 + 1 columns, no PML
    ((92, 124, 28), 8, 1),
])
def test_adjoint_and_small_forward(shape, pml, nrhs):
    hz, s = _solver(shape, pml, nrhs)
    for level in range(3):
        x = torch.from_numpy(W.random_complex((nrhs,) + s.level_shape[level], 3)).to("cuda", torch.complex64)
        y = torch.from_numpy(W.random_complex(x.shape, 4)).to("cuda", torch.complex64)
        x128, y128 = x.to(torch.complex128), y.to(torch.complex128)
        pairs = [(hz.HZ_OP_A, hz.HZ_OP_A_ADJ), (hz.HZ_OP_B, hz.HZ_OP_B_ADJ)]
        for op, adj in pairs + ([(hz.HZ_OP_Q, hz.HZ_OP_Q_ADJ)] if level == 0 else []):
            Ax = s.iofd_apply(x128, op=op, level=level)
            Ay = s.iofd_apply(y128, op=adj, level=level)
            d = torch.vdot(y128.reshape(-1), Ax.reshape(-1)) - torch.vdot(Ay.reshape(-1), x128.reshape(-1))
            n = torch.linalg.vector_norm(Ax) * torch.linalg.vector_norm(y128)
            assert float(abs(d) / n) <= TOL128
            assert _rel(s.iofd_apply(x, op=op, level=level), Ax) <= TOL64
            assert _rel(s.iofd_apply(y, op=adj, level=level), Ay) <= TOL64
        r, n2 = s.residual_static(y128, x128, level=level)
        assert _rel(r, y128 - s.iofd_apply(x128, level=level)) <= TOL128
        assert torch.allclose(n2, (r.abs() ** 2).flatten(1).sum(1) if nrhs > 1 else (r.abs() ** 2).sum(), rtol=1e-12)
        assert _rel(s.iofd_jacobi(x, level=level), s.iofd_jacobi(x128, level=level)) <= TOL64
    s.close()


@pytest.mark.parametrize("rows", [2, 3, 5])
def test_coarse_weight_tables(rows):
    """Tables of few rows: wide segments, so more parts per segment for the cubics."""
    import paper_2608_22946_gb300 as hz_
    t = hz_.load_table()
    t = np.ascontiguousarray(t[np.linspace(0, len(t) - 1, rows).astype(int)])
    hz, s = _solver((84, 84, 84), 4, 1, table=t)  # 6.1e5 nodes: the march
    x = torch.from_numpy(W.random_complex((1,) + s.level_shape[0], 3)).to("cuda", torch.complex64)
    for op in (hz.HZ_OP_A, hz.HZ_OP_B):
        assert _rel(s.iofd_apply(x, op=op), s.iofd_apply(x.to(torch.complex128), op=op)) <= TOL64
    s.close()
