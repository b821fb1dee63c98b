"""The single-precision march (csrc/hz_march.cuh) against the complex128 kernels.

Grids on its edges: cores one column short of, equal to and past a 64-column
tile, no PML (element-wise copies, zero halo), an even-sized level (no two-row
pitch for the tensor copies), one to three right-hand sides (one and two per
block), fields that start on an odd 8-byte boundary, and z-windows.

Tolerance: a row sums 27 products of single-precision weights, each a few
roundings from its exact value: at most about 40 u sum |w||x| per row with
u = 6e-8, and sum |w||x| is two to three times |row| in the root mean square.
2e-6 of the L2 norm is a third of that worst case.
"""
import numpy as np
import pytest

import hz_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 2e-6


def _solver(shape, pml, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    rng = np.random.default_rng(5)
    nx, ny, nz = shape
    c = 1.5 + rng.random((nz + 1, ny + 1, nx + 1))
    h, omega = W.grid_params(min(shape), pml, 1.5)
    return hz, hz.Solver(shape, pml, h, omega, c, params=hz.default_params(autotune=0), max_nrhs=nrhs)


def _rel(a, b):
    return float(torch.linalg.vector_norm(a.to(torch.complex128) - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("shape,pml,level,nrhs", [
    ((72, 136, 212), 4, 0, 1),     # core 63 x 127
    ((76, 144, 100), 4, 0, 2),     # core 67 x 135, two right-hand sides per block
    ((140, 76, 100), 8, 0, 3),     # three: one per block
    ((88, 84, 140), 0, 0, 2),      # no PML
    ((260, 256, 252), 8, 1, 1),    # 2h level
    ((324, 324, 324), 8, 2, 2),    # 82^3: even-sized level (its Jacobi map and residual: gather form)
    ((300, 300, 24), 4, 0, 1),     # few core planes
])
def test_march_matches_complex128(shape, pml, level, nrhs):
    hz, s = _solver(shape, pml, nrhs)
    x = torch.from_numpy(W.random_complex((nrhs,) + s.level_shape[level], 3)).to("cuda", torch.complex64)
    g = torch.from_numpy(W.random_complex(x.shape, 4)).to("cuda", torch.complex64)
    x128, g128 = x.to(torch.complex128), g.to(torch.complex128)
    odd = torch.empty(x.numel() + 1, dtype=torch.complex64, device="cuda")[1:].view(x.shape)  # 8 mod 16
    odd.copy_(x)
    for op in ([hz.HZ_OP_A, hz.HZ_OP_B] + ([hz.HZ_OP_Q] if level == 0 else [])):
        ref = s.iofd_apply(x128, op=op, level=level)
        assert _rel(s.iofd_apply(x, op=op, level=level), ref) <= TOL
        assert torch.equal(s.iofd_apply(odd, op=op, level=level), s.iofd_apply(x, op=op, level=level))
    for op in (hz.HZ_OP_A, hz.HZ_OP_B):
        ref, n2 = s.residual_static(g128, x128, op=op, level=level)
        r, m2 = s.residual_static(g, x, op=op, level=level)
        assert _rel(r, ref) <= TOL and torch.allclose(m2, n2, rtol=1e-5, atol=0)
    assert _rel(s.iofd_jacobi(x, level=level), s.iofd_jacobi(x128, level=level)) <= TOL
    assert _rel(s.iofd_jacobi(odd, level=level), s.iofd_jacobi(x128, level=level)) <= TOL
    s.close()


@pytest.mark.parametrize("z0,z1", [(0, 7), (5, 40), (33, 61)])
def test_march_window_equals_the_whole_grid(z0, z1):
    hz, s = _solver((72, 136, 60), 4, 2)  # 2^19 nodes: the march
    x = torch.from_numpy(W.random_complex((2,) + s.level_shape[0], 9)).to("cuda", torch.complex64)
    pad = torch.zeros((2, 63, 137, 73), dtype=torch.complex64, device="cuda")
    pad[:, 1:62] = x
    y = s.iofd_apply_window(pad[:, z0:z1 + 2].contiguous(), z0, z1)
    assert _rel(y, s.iofd_apply(x)[:, z0:z1].to(torch.complex128)) <= 1e-7
    s.close()


@pytest.mark.parametrize("nJ", [3])
def test_further_jacobi_sweeps(nJ):
    """The preconditioner with three sweeps on every level (the single-sweep kernel)."""
    hz, s = _solver((132, 132, 132), 4, 1)
    p = hz.default_params(autotune=0, nJ_h=nJ, nJ_2h=nJ, nJ_4h=nJ)
    s.close()
    c = 1.5 + np.random.default_rng(5).random((133, 133, 133))
    h, omega = W.grid_params(132, 4, 1.5)
    s = hz.Solver(132, 4, h, omega, c, params=p)
    r = torch.from_numpy(W.random_complex(s.level_shape[0], 11)).to("cuda", torch.complex64)
    assert _rel(s.threegrid_precond(r), s.threegrid_precond(r.to(torch.complex128))) <= 2e-4
    s.close()
