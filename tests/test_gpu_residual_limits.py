"""iofd_residual_static near and past the 65,536 partial sums of its scratch.

257 x 257 x 69 nodes and 64 right-hand sides: 65,664 blocks of the complex128
launch at its heuristic z-blocks (hz_layout_check), so the norm is a pass of its
own; 65 planes fit.  The call takes both, in both precisions.

Tolerances: the norm sums |r|^2 over 4.6 million nodes in the fields' precision per
thread and in FP64 across threads: at most a few hundred additions in a row, each
off by u/2 relative, which is 1e-5 for complex64 (u = 1.2e-7) and 3e-14 for
complex128.  Residuals as in test_gpu_march.py.
"""
import pytest

import hz_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [64, 68])
def test_residual_past_the_static_scratch(nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    shape, pml, nrhs = (256, 256, nz), 8, 64
    _, blocks, bad = hz.layout_check(shape, pml, nrhs=nrhs)
    assert bad == 0 and (blocks * nrhs > 65536) == (nz == 68)
    h, omega = W.grid_params(nz, pml, 1.5)
    c = 1.5 + torch.rand((nz + 1, 257, 257), dtype=torch.float64, device="cuda",
                         generator=torch.Generator("cuda").manual_seed(3))
    s = hz.Solver(shape, pml, h, omega, c, params=hz.default_params(autotune=0), max_nrhs=nrhs)
    gen = torch.Generator("cuda").manual_seed(4)
    for dt, tol, ntol in ((torch.complex64, 2e-6, 1e-5), (torch.complex128, 3e-14, 3e-14)):
        x = torch.randn((nrhs, nz + 1, 257, 257), dtype=dt, device="cuda", generator=gen)
        g = torch.randn(x.shape, dtype=dt, device="cuda", generator=gen)
        r, n2 = s.residual_static(g, x)
        for k in (0, 1, nrhs - 1):
            ref = g[k].to(torch.complex128) - s.iofd_apply(x[k].to(torch.complex128))
            assert float(torch.linalg.vector_norm(r[k] - ref) / torch.linalg.vector_norm(ref)) <= tol
        ref2 = torch.stack([(r[k].to(torch.complex128).abs() ** 2).sum() for k in range(nrhs)])
        assert torch.allclose(n2, ref2, rtol=ntol, atol=0)
        del x, g, r
    s.close()


def test_complex128_residual_on_two_streams():
    """105^3 in complex128: rectangle and PML frame are two launches, the frame on the
    handle's second stream, and both add their block sums to the one static array."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_22946_gb300 as hz
    w = W.layered_inclusion(n=104, n_pml=8, nsrc=1)
    s = hz.Solver(w.n, w.n_pml, w.h, w.omega, w.c, max_nrhs=2)
    gen = torch.Generator("cuda").manual_seed(5)
    for _ in range(2):
        x = torch.randn((2,) + s.level_shape[0], dtype=torch.complex128, device="cuda", generator=gen)
        g = torch.randn(x.shape, dtype=torch.complex128, device="cuda", generator=gen)
        r, n2 = s.residual_static(g, x)
        ref = g - s.iofd_apply(x)
        assert float(torch.linalg.vector_norm(r - ref) / torch.linalg.vector_norm(ref)) <= 3e-14
        assert torch.allclose(n2, (ref.abs() ** 2).flatten(1).sum(1), rtol=3e-14, atol=0)
    s.close()
