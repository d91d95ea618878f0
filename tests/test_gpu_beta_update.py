"""A beta field updated in place and given to init_domain again: what the set-up
keeps of it (diagonal, spectrum bounds, sign, face means in adjoint contexts) is
that of the new values, to the bit of a fresh context's results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2209_15095_gb300 import build

    build.build()
    from paper_2209_15095_gb300 import etd

    return etd


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ndim,n", [(2, 33), (3, 20)])
def test_update_in_place(lib, ndim, n, precision, adjoint):
    x = np.meshgrid(*([np.linspace(-1.6, 1.6, n)] * ndim), indexing="ij")
    r = np.sqrt(sum(c * c for c in x))
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    phi, u = dev(r - 1.0), dev(np.where(r < 0.9, np.cos(r), 0.0))
    s = np.sin(1.7 * x[0] + 0.4)
    fields = [1.0 + 0.3 * s, 0.1 + 0.3 * s, 0.8 - 0.2 * s, None, 1.0 + 0.3 * s]  # the second: negative in places

    def context():
        return lib.Context((n,) * ndim, (-1.6,) * ndim, (1.6,) * ndim, precision=precision, tol=1e-9, m_max=40,
                           reaction="logistic_ak", rparams=(1.0, 1.0), adjoint=adjoint)

    def results(ctx, beta):
        ctx.init_domain(0, phi, beta)
        out = [torch.zeros_like(u) for _ in range(2)]
        ctx.step_explicit(0, 0.01, u, u, out[0])
        ctx.apply_operator(0, 1.0, u, out[1])
        if adjoint:
            lam, acc, gb = u.clone(), torch.zeros_like(u), torch.zeros_like(u)
            gp = torch.zeros(1, dtype=torch.float64, device="cuda")
            ctx.adjoint_step(0, 0.01, u, u, True, lam, acc, gb, gp)
            out += [lam, gp]
        ctx.sync()
        return out

    ctx = context()
    field = torch.zeros_like(u)
    for f in fields:
        if f is not None:
            field.copy_(dev(f))
        got = results(ctx, None if f is None else field)
        want = results(context(), None if f is None else dev(f))
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        assert got[0].abs().max() > 0.1
