"""The Poisson solve on both sides of the point count where the search direction gets a
pass of its own (3 to 8 points per thread, by dimension and kind of beta):
the true residual of the solution, by etd_apply_operator, and the iteration count
against the grid's spacing (conjugate gradients take about as many iterations as
the domain has nodes across, whichever form)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("ndim,n", [(2, 700), (2, 1400), (3, 100), (3, 140), (4, 40), (4, 56)])
def test_true_residual(ndim, n, field):
    from paper_2209_15095_gb300 import build

    build.build()
    from paper_2209_15095_gb300 import etd

    x = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda")
    ax = [x.view([-1 if i == d else 1 for i in range(ndim)]) for d in range(ndim)]
    r = sum(a * a for a in ax).sqrt()
    phi = (r - 0.7).contiguous()
    beta = (1.0 + 0.3 * torch.sin(3.0 * ax[0]) * torch.cos(2.0 * ax[1])).expand((n,) * ndim).contiguous()
    f = (1.0 + 0.5 * torch.cos(4.0 * r + ax[0])).contiguous()
    ctx = etd.Context((n,) * ndim, (-1.0,) * ndim, (1.0,) * ndim, m_max=5)
    ctx.init_domain(0, phi, beta if field else None)
    u = torch.zeros_like(phi)
    tol = 1e-9
    it, res = ctx.poisson_solve(0, f, u, tol=tol)
    assert res <= tol and n // 4 < it < 6 * n
    cu = torch.zeros_like(phi)
    ctx.apply_operator(0, 1.0, u, cu)
    ctx.sync()
    kind = ctx.read_domain(0)["kind"] & 3
    comp = torch.tensor(np.asarray(kind) == 2, device="cuda")
    true = torch.linalg.norm((cu - f)[comp]) / torch.linalg.norm(f[comp])
    # the recurrence drifts from the true residual by the rounding of u, 2^-53 |C| |u| / |f|
    drift = 2.0 ** -50 * 4 * ndim * 1.3 * (n - 1) ** 2 / 4 * torch.linalg.norm(u[comp]) / torch.linalg.norm(f[comp])
    assert true <= tol + drift
