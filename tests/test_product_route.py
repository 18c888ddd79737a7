"""Which FP64 and double-float lists run on the digit-sliced products (CPU: contexts only).

The digits' time has a part per product whatever its size, the CUDA cores' goes with the multiply-adds: lists of
few channels belong on the CUDA cores from some lattice size on, all 52 or 90 channels never do."""
import pytest

from paper_1510_00903_gb300 import bbc


def _digits(precision, L, chans):
    ctx = bbc.bbc_create(L, 4, 0, 0.3, 0.4, precision, chans)
    try:
        return bbc.bbc_digit_products(ctx)
    finally:
        bbc.bbc_destroy(ctx)


@pytest.mark.parametrize("L", [2, 4, 8, 16, 24, 32, 48])
@pytest.mark.parametrize("precision", [bbc.BBC_FP64, bbc.BBC_DF64])
def test_whole_lists_and_small_lattices(precision, L):
    assert _digits(precision, L, list(range(52))) and _digits(precision, L, list(range(64, 154)))
    if L <= 8:
        assert all(_digits(precision, L, [c]) for c in (0, 1, 14, 51, 64, 99))


@pytest.mark.parametrize("precision", [bbc.BBC_FP64, bbc.BBC_DF64])
@pytest.mark.parametrize("chans", [[51], [64], [99], [79, 120, 149], bbc.DELTA_DELTA[:4]])
def test_few_channels_on_large_lattices(precision, chans):
    route = [_digits(precision, L, chans) for L in (2, 4, 8, 16, 24, 32, 48)]
    assert route == sorted(route, reverse=True)  # one line between the two
    if precision == bbc.BBC_DF64:  # (FP64: the pipe is narrow, three or four channels may stay on the digits)
        assert not any(route[4:])


def test_other_precisions_and_plans_not_held():
    assert not _digits(bbc.BBC_MIXED_FP32, 4, list(range(52)))
    assert not _digits(bbc.BBC_FP64, 4, list(range(52)) + [64])  # more trace blocks than a set holds
    assert not _digits(bbc.BBC_FP64, 4, [150])
