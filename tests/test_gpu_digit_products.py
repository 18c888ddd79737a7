"""GPU tests of the digit-sliced products on inputs that strain them.

Tolerance: the 1e-12 of the FP64-accurate paths (relative to the channel's
maximum), as in test_gpu_exact_products.py."""
import pytest

torch = pytest.importorskip("torch")

import oracle.oracle as orc  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def bbc():
    from paper_1510_00903_gb300 import bbc as m
    return m


def _run(bbc, L, Sl, Ss, chans, precision, lower=False):
    cor = bbc.Correlators(L, 4, 0, 0.3, 0.4, channels=chans, precision=precision,
                          components=bbc.BBC_LOWER if lower else bbc.BBC_UPPER)
    Sl, Ss = (torch.as_tensor(S).to(cor.device)[None] for S in (Sl, Ss))
    out = cor.run(Sl, Ss, [0], normalised=False)[0]
    cor.status()
    cor.close()
    return out


def _oracle(L, Sl, Ss, chans, lower=False):
    Sl, Ss = (torch.as_tensor(S).cpu().numpy() for S in (Sl, Ss))
    return torch.from_numpy(orc.correlator(L, Sl, Sl, Ss, chans, lower=lower)).cuda()


def _err(got, want):
    """Per channel, relative to the channel's maximum; the largest of them."""
    return ((got - want).abs().flatten(1).amax(1) / want.abs().flatten(1).amax(1)).max().item()


def _normal(gen, shape):
    return torch.randn(shape, generator=gen, dtype=torch.complex128, device="cuda")


@pytest.mark.parametrize("eps", [0.3, 0.1, 0.03, 1e-3])
@pytest.mark.parametrize("L", [8, 16, 24, 32, 48])
def test_smooth_fields_in_double_float(bbc, L, eps):
    """A constant part and eps times noise: at q != 0 every block is a difference of large equal terms, and the
    high words of its double-float pairs cancel in the forward transform.  L = 8 against the oracle, larger
    lattices, all octet channels, against the FP64 path."""
    gen = torch.Generator(device="cuda").manual_seed(17 * L)
    Sl, Ss = (torch.eye(12, device="cuda") + 0.1 * _normal(gen, (1, 12, 12)) + eps * _normal(gen, (L ** 3, 12, 12))
              for _ in range(2))
    chans = [0, 16] if L == 8 else list(range(52))
    want = _oracle(L, Sl, Ss, chans) if L == 8 else _run(bbc, L, Sl, Ss, chans, bbc.BBC_FP64)
    assert _err(_run(bbc, L, Sl, Ss, chans, bbc.BBC_DF64), want) <= TOL


@pytest.mark.parametrize("w", [0.1, 1e-2, 1e-5])
@pytest.mark.parametrize("lower", [False, True])
@pytest.mark.parametrize("chans", [[0, 1, 10, 16, 51], [70, 99, 145, 150]])
@pytest.mark.parametrize("precision", [0, 3])
def test_graded_dirac_components(bbc, precision, chans, lower, w):
    """Lower or upper Dirac components w times the other ones, of the source index alone and of both indices:
    slices of a block that are far smaller than the block."""
    L, gen = 4, torch.Generator(device="cuda").manual_seed(8)
    g = torch.tensor([1.0] * 6 + [w] * 6, device="cuda", dtype=torch.float64)
    one = torch.ones_like(g)
    for sink, src in ((one, g), (g, g), (one, g.flip(0)), (g.flip(0), g.flip(0))):
        Sl, Ss = (_normal(gen, (L ** 3, 12, 12)) * (sink[:, None] * src) for _ in range(2))
        want = _oracle(L, Sl, Ss, chans, lower)
        assert _err(_run(bbc, L, Sl, Ss, chans, precision, lower), want) <= TOL
