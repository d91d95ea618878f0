"""The word-parallel classification on grids whose rows are not whole 32-node
words: rows of 8 to 101 nodes (up to five rows in a word), sizes that leave a
partial last word; random-sign interiors against the per-node definition, the
margin error, and a shrinking domain whose vector entries have to be zeroed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [(40, 33), (9, 8), (57, 101), (12, 11, 10), (17, 16, 48), (31, 33, 35), (9, 10, 11, 12), (12, 12, 12, 48)]


def _ctx(shape):
    from paper_2209_15095_gb300 import build

    build.build()
    from paper_2209_15095_gb300 import etd

    h = 0.01
    return etd.Context(shape, [0.0] * len(shape), [h * (n - 1) for n in shape], reaction="none", m_max=10)


def _reference(phi):
    inside = phi < 0
    comp = inside.copy()
    for d in range(phi.ndim):
        for s in (-1, 1):
            nb = np.roll(inside, s, axis=d)
            edge = [slice(None)] * phi.ndim
            edge[d] = 0 if s == 1 else -1
            nb[tuple(edge)] = False
            comp &= nb
    return inside.astype(np.uint8) + comp.astype(np.uint8)


def _random_phi(shape, rng, p):
    phi = np.where(rng.random(shape) < p, -1.0, 1.0)
    core = np.full(shape, False)
    core[tuple(slice(3, n - 3) for n in shape)] = True
    return np.where(core, phi, 1.0)


@pytest.mark.parametrize("shape", SHAPES)
def test_kinds(shape):
    rng = np.random.default_rng(7)
    ctx = _ctx(shape)
    for p in (0.3, 0.95, 1.0, 0.0):  # the same context: the domain grows, then empties
        phi = _random_phi(shape, rng, p)
        ctx.init_domain(0, torch.tensor(phi, device="cuda"))
        dom = ctx.read_domain(0)
        ref = _reference(phi)
        np.testing.assert_array_equal(dom["kind"] & 3, ref)
        np.testing.assert_array_equal(dom["idx"], np.flatnonzero(ref.ravel() == 2))


@pytest.mark.parametrize("shape", SHAPES)
def test_margin_error(shape):
    from paper_2209_15095_gb300 import etd

    ctx = _ctx(shape)
    for d in range(len(shape)):
        for at in (0, 2, shape[d] - 3, shape[d] - 1):
            phi = np.ones(shape)
            node = [n // 2 for n in shape]
            node[d] = at
            phi[tuple(node)] = -1.0
            ctx.init_domain(0, torch.tensor(phi, device="cuda"))
            with pytest.raises(etd.EtdError, match="ETD_ERR_DOMAIN"):
                ctx.sync()
        for at in (3, shape[d] - 4):
            phi = np.ones(shape)
            node = [n // 2 for n in shape]
            node[d] = at
            phi[tuple(node)] = -1.0
            ctx.init_domain(0, torch.tensor(phi, device="cuda"))
            ctx.sync()


@pytest.mark.parametrize("shape", [(57, 101), (31, 33, 35)])
def test_shrunk_domain(shape):
    """A combination on a domain that has shrunk equals one in a new context
    bit for bit: no entry of the larger domain is left in the stencil's reach."""
    ax = np.meshgrid(*[np.arange(n) - 0.5 * (n - 1) for n in shape], indexing="ij")
    r = np.sqrt(sum(a * a for a in ax))
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    v = [dev(np.cos(0.1 * r) * (k + 1)) for k in range(3)]
    big, small = dev(r - 0.5 * min(shape) + 5.0), dev(r - 0.3 * min(shape))
    out = []
    for first in (big, small):
        ctx = _ctx(shape)
        y = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for phi in (first, small):
            ctx.init_domain(0, phi)
            y.zero_()
            ctx.phi_combination(0, 1e-5, *v, y)
        ctx.sync()
        out.append(y.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
