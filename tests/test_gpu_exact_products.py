"""GPU tests of the digit-sliced tensor-core products of the FP64-accurate
paths: operand counts that leave ragged tiles (one channel: 12 blocks, a few,
all 64 octet ids: 48 blocks; decuplet ids: same-orientation traces and
transposed slices), small lattices (fewer pairs than SMs, q = -q
only), rows of very different size, zero and non-finite propagators.

Tolerance: the 1e-12 of the FP64-accurate paths (relative to the channel's
maximum).  A row value keeps 2^-55 of its row's largest magnitude and the sums
are exact, so even rows whose components differ by 1e3 stay far inside it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.oracle as orc  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def bbc():
    from paper_1510_00903_gb300 import bbc as m
    return m


def _run(bbc, L, Sl, Ss, chans, precision, lower=False):
    cor = bbc.Correlators(L, 4, 0, 0.3, 0.4, channels=chans, precision=precision,
                          components=bbc.BBC_LOWER if lower else bbc.BBC_UPPER)
    dev = cor.device
    out = cor.run(torch.from_numpy(Sl).to(dev)[None], torch.from_numpy(Ss).to(dev)[None], [0], normalised=False)
    cor.status()
    got = out[0].cpu().numpy()
    cor.close()
    return got


def _check(got, want, vanish=()):
    """vanish: positions of channels that are identically zero in the isospin limit (their oracle values are
    rounding errors of the same sums): held to the scale of the other channels."""
    scale = np.abs(want).reshape(want.shape[0], -1).max(axis=1)
    scale[list(vanish)] = scale.max()
    err = np.abs(got - want).reshape(want.shape[0], -1).max(axis=1)
    assert (err <= TOL * scale).all(), (err / scale).max()


@pytest.mark.parametrize("precision", [0, 3])
@pytest.mark.parametrize("L,chans,lower", [(2, [0], False), (2, list(range(64)), False), (4, [1, 2], True),
                                           (4, [11, 20, 51], False), (4, list(range(52)), False),
                                           (4, [64, 70, 99, 143, 145, 150], False), (2, list(range(145, 154)), True)])
def test_operand_counts(bbc, precision, L, chans, lower):
    F = synth.flavour_set(L, 4, 0, 0.3, 0.4, seed=90 + L, times=[0])
    want = orc.correlator(L, F["u"][0], F["u"][0], F["s"][0], chans, lower=lower)
    _check(_run(bbc, L, F["u"][0], F["s"][0], chans, precision, lower), want,
           [i for i, c in enumerate(chans) if 52 <= c <= 55])


@pytest.mark.parametrize("precision", [0, 3])
def test_rows_of_very_different_size(bbc, precision):
    """Lower Dirac components a thousandth of the upper ones, the strange quark 1e-8 of the light one."""
    L, chans = 4, [0, 1, 10, 16, 51]
    F = synth.flavour_set(L, 4, 0, 0.3, 0.4, seed=95, times=[0])
    w = np.array([1.0] * 6 + [1e-3] * 6)
    Sl = F["u"][0] * (w[:, None] * w[None, :])
    Ss = F["s"][0] * (w[:, None] * w[None, :]) * 1e-8
    want = orc.correlator(L, Sl, Sl, Ss, chans)
    _check(_run(bbc, L, Sl, Ss, chans, precision), want)


@pytest.mark.parametrize("precision", [0, 3])
def test_zero_and_non_finite(bbc, precision):
    """Zero strange propagators give exact zeros where a strange quark takes part; an infinite light entry
    spoils every channel (each reads the light quark at every q), never silently."""
    L, chans = 4, [0, 1, 51]
    F = synth.flavour_set(L, 4, 0, 0.3, 0.4, seed=96, times=[0])
    Sl, zero = F["u"][0], np.zeros_like(F["s"][0])
    got = _run(bbc, L, Sl, zero, chans, precision)
    _check(got[:1], orc.correlator(L, Sl, Sl, zero, chans[:1]))
    assert (got[1:] == 0).all()
    bad = Sl.copy()
    bad[5, 3, 4] = np.inf
    assert not np.isfinite(_run(bbc, L, bad, F["s"][0], chans, precision)).any(axis=(1, 2)).all()
