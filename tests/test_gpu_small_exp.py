"""The Chebyshev series of the small exponential (the Krylov error check) over
the sizes and spectra where it changes form: one or two rows per lane (m + 3
above 32), a below 1 up to above 512 (several steps), p = 2 and 3; and a beta
field with negative values, which takes the Gershgorin interval.  The phi-
combination against a dense eigen-decomposition: the Krylov tolerance times
its safety margin of 20 (as for the oracle's own Krylov routine), relative to
the largest of |v_0|, |v_1|, |v_2|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _phi(k, z):
    """phi_k of real z by its definition; the series where that cancels."""
    z = np.asarray(z, dtype=np.longdouble)
    small = np.abs(z) < 1.0
    zs, zl = np.where(small, z, 0), np.where(small, 1, z)
    t = np.ones_like(z)
    for j in range(1, k + 1):
        t = t / j
    ser = np.zeros_like(z)
    for i in range(40):
        ser = ser + t
        t = t * zs / (i + k + 1)
    f, fact = np.exp(zl), np.longdouble(1)
    for j in range(k):
        f = (f - 1 / fact) / zl
        fact = fact * (j + 1)
    return np.where(small, ser, f).astype(np.float64)


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("m_max", [5, 29, 30, 60])
@pytest.mark.parametrize("rho", [0.5, 60.0, 3000.0])
@pytest.mark.parametrize("negative", [False, True])
def test_phi_combination_spectra(rho, m_max, p, negative):
    from oracle.eb import EBOperator
    from oracle.grid import Grid
    from paper_2209_15095_gb300 import build

    build.build()
    from paper_2209_15095_gb300 import etd

    n, box, tol = 26, 1.0, 1e-9
    g = Grid((n, n), (-box,) * 2, (box,) * 2)
    x = g.coords()
    phi = np.sqrt(x[0] ** 2 + x[1] ** 2) - 0.8
    beta = 1.0 + 0.3 * np.sin(3 * x[0]) * np.cos(2 * x[1])
    if negative:
        beta = np.where((np.abs(x[0]) < 0.1) & (np.abs(x[1] - 0.2) < 0.1), -0.02, beta)
        rho = min(rho, 60.0)  # the growing modes stay representable
    op = EBOperator(g, phi, beta)
    C = op.C.toarray()
    lam, Q = np.linalg.eigh(0.5 * (C + C.T))
    dt = rho / np.abs(lam).max()
    rng = np.random.default_rng(5)
    v = [rng.standard_normal(op.ncomp) for _ in range(p + 1)]
    ref = sum(Q @ (_phi(k, dt * lam) * (Q.T @ v[k])) for k in range(p + 1))
    ctx = etd.Context(g.n, g.lo, g.hi, tol=tol, m_max=m_max, reaction="none")
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    ctx.init_domain(0, dev(phi), dev(beta))
    y = torch.zeros(g.n, dtype=torch.float64, device="cuda")
    vs = [dev(op.to_grid(a)) for a in v]
    (ctx.phi_combination if p == 2 else ctx.phi_combination3)(0, dt, *vs, y)
    ctx.sync()
    scale = max(np.linalg.norm(a) for a in v + [ref])
    assert np.linalg.norm(op.from_grid(y.cpu().numpy()) - ref) <= 20 * tol * scale
