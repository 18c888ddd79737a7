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


# (double-float has FP32's range: a block of three quarks of 1e-20 underflows in its arithmetic)
@pytest.mark.parametrize("precision,w", [(0, 1e-2), (0, 1e-4), (0, 1e-20), (3, 1e-2), (3, 1e-4)])
@pytest.mark.parametrize("lower", [False, True])
def test_flavours_graded_against_each_other(bbc, precision, lower, w):
    """Light quarks from upper, strange quarks from lower Dirac components: the large values of one row meet the
    small ones of the other, and products lie far below what their rows' maxima suggest."""
    L, chans, gen = 4, [0, 1, 10, 16, 51, 70, 145, 150], torch.Generator(device="cuda").manual_seed(9)
    g = torch.tensor([1.0] * 6 + [w] * 6, device="cuda", dtype=torch.float64)
    for gl, gs in ((g, g.flip(0)), (g.flip(0), g)):
        Sl, Ss = _normal(gen, (L ** 3, 12, 12)) * gl, _normal(gen, (L ** 3, 12, 12)) * gs
        assert _err(_run(bbc, L, Sl, Ss, chans, precision, lower), _oracle(L, Sl, Ss, chans, lower)) <= TOL


@pytest.mark.parametrize("chans", [list(range(52)), list(range(64, 154, 7))])
@pytest.mark.parametrize("precision", [0, 3])
def test_products_that_vanish_term_by_term(bbc, precision, chans):
    """Propagators diagonal in colour (unit gauge links): most terms of every product are exact zeros."""
    L, gen = 4, torch.Generator(device="cuda").manual_seed(10)
    Sl, Ss = (torch.einsum("vab,cd->vacbd", _normal(gen, (L ** 3, 4, 4)),
                           torch.eye(3, dtype=torch.complex128, device="cuda")).reshape(L ** 3, 12, 12).contiguous()
              for _ in range(2))
    want = _oracle(L, Sl, Ss, chans)
    scale = want.abs().amax()
    got = _run(bbc, L, Sl, Ss, chans, precision)
    live = want.abs().flatten(1).amax(1) > 1e-9 * scale
    assert live.any() and _err(got[live], want[live]) <= TOL
    assert ((got - want)[~live].abs() <= TOL * scale).all()


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("precision", [0, 3])
def test_non_finite_values_reach_what_reads_them(bbc, precision, value):
    """A non-finite light entry spoils every channel, a strange one those with strange quarks and no other."""
    L, chans, gen = 4, [0, 1, 16, 51], torch.Generator(device="cuda").manual_seed(11)
    Sl, Ss = (_normal(gen, (L ** 3, 12, 12)) for _ in range(2))
    bad = [S.clone() for S in (Sl, Ss)]
    for S in bad:
        S[5, 3, 4] = value
    got = _run(bbc, L, bad[0], Ss, chans, precision)
    assert (~torch.isfinite(torch.view_as_real(got))).flatten(1).any(1).all()
    got = _run(bbc, L, Sl, bad[1], chans, precision)
    assert (~torch.isfinite(torch.view_as_real(got[1:]))).flatten(1).any(1).all()
    assert _err(got[:1], _oracle(L, Sl, Ss, chans[:1])) <= TOL


@pytest.mark.parametrize("chans", [[0], list(range(52)), [64, 70, 99, 145]])
@pytest.mark.parametrize("precision", [0, 3])
def test_products_waits_run_out_and_the_context_recovers(bbc, precision, chans):
    """With one poll per wait the first waits give up: the kernel records it, frees its tensor memory and returns,
    and the context stays usable."""
    L, gen = 4, torch.Generator(device="cuda").manual_seed(12)
    Sl, Ss = (_normal(gen, (1, L ** 3, 12, 12)) for _ in range(2))
    cor = bbc.Correlators(L, 4, 0, 0.3, 0.4, channels=chans, precision=precision)
    assert bbc.bbc_check_products_wait(cor.ctx, 1) == bbc.BBC_ESTATE  # nothing built
    before = cor.run(Sl, Ss, [0]).clone()
    cor.status()
    for _ in range(3):
        assert bbc.bbc_check_products_wait(cor.ctx, 1) == bbc.BBC_ETIMEOUT
        assert "bounded wait" in bbc.lib().bbc_last_error(cor.ctx).decode()
    cor.status()  # the record was read and cleared
    assert bbc.bbc_check_products_wait(cor.ctx, 1 << 22) == bbc.BBC_OK
    assert torch.equal(cor.run(Sl, Ss, [0]), before)
    cor.status()
    cor.close()


def test_products_wait_self_test_needs_the_digit_products(bbc):
    cor = bbc.Correlators(4, 4, 0, 0.3, 0.4, channels=[0], precision=bbc.BBC_MIXED_FP32)
    assert bbc.bbc_check_products_wait(cor.ctx, 1) == bbc.BBC_ESTATE
    assert bbc.bbc_check_products_wait(cor.ctx, 0) == bbc.BBC_EINVAL
    cor.close()


@pytest.mark.parametrize("precision,L,few,many", [(0, 24, [51], range(10, 52)), (0, 24, [64], range(64, 154)),
                                                  (3, 16, [14], range(10, 52)), (3, 24, [64], range(64, 154)),
                                                  (3, 32, [0, 51], range(52)), (3, 48, [51], range(10, 52))])
def test_few_channels_on_the_cuda_cores_agree_with_the_digits(bbc, precision, L, few, many):
    """The same channels from a list short enough for the CUDA cores and from one on the digit products."""
    gen = torch.Generator(device="cuda").manual_seed(13 + L)
    Sl, Ss = (_normal(gen, (L ** 3, 12, 12)) for _ in range(2))
    many, routes = list(many), []
    for chans in (few, many):
        ctx = bbc.bbc_create(L, 4, 0, 0.3, 0.4, precision, chans)
        routes.append(bbc.bbc_digit_products(ctx))
        bbc.bbc_destroy(ctx)
    assert routes == [False, True]
    got, want = _run(bbc, L, Sl, Ss, few, precision), _run(bbc, L, Sl, Ss, many, precision)
    assert _err(got, want[[many.index(c) for c in few]]) <= TOL
