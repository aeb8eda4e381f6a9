"""The division-free rounding of the resolve kernel (round_quotient2) against
the rule it stands for, floor(RN(RN(X / Z) + 0.5)), emulated step by step: every
quotient that it calls settled must give the rule's integer, for any reciprocal
within a few last places, and the quotients it leaves to the division must be
few."""
import numpy as np
import pytest

F = np.float32


def _rule(X, Z):
    return np.floor(F(X / Z) + F(0.5)).astype(np.int64)


def _settled(X, Z, ulps, dim):
    """(integer, settled) with a reciprocal `ulps` last places off."""
    k = int(np.ceil(np.log2(dim))) if dim > 1 else 0
    eps = F(2.0 ** (k - 25)) + F(2.0 ** -20)
    r = (F(1) / Z) * F(1 + ulps * 2.0 ** -23)
    Xd, Zd, rd = X.astype(np.float64), Z.astype(np.float64), r.astype(np.float64)
    m = np.floor(Xd * rd)                                   # the product of two floats is exact in 64 bits
    f = (Xd - m * Zd).astype(F)                             # the fused operation's one rounding
    phi = f.astype(np.float64) * rd
    near = (phi - 0.5).astype(F)
    return (m + np.rint(phi)).astype(np.int64), np.abs(near) > eps


@pytest.mark.parametrize("dim", [1, 2, 3, 200, 1280, 1920, 8192, 1 << 20])
@pytest.mark.parametrize("ulps", [-3, -1, 0, 1, 3])
def test_settled_quotients_round_like_the_division(dim, ulps):
    rng = np.random.default_rng(100 + dim + ulps)
    n = 200000
    Z = F(10.0 ** rng.uniform(-3, 6, n))
    q = rng.uniform(-2, dim + 2, n)
    X = F(q * Z)
    # half of them beside a rounding boundary: (integer + 1/2) Z and a few last places around
    half = n // 2
    base = rng.integers(-1, dim + 1, half) + 0.5
    Xh = F(base * Z[:half].astype(np.float64))
    for _ in range(3):
        Xh = np.where(rng.random(half) < 0.5, np.nextafter(Xh, F(np.inf)), np.nextafter(Xh, F(-np.inf)))
    X[:half] = Xh
    got, ok = _settled(X, Z, ulps, dim)
    want = _rule(X, Z)
    inside = (want >= 0) & (want < dim) | (got >= 0) & (got < dim)
    bad = ok & inside & (got != want)
    assert not bad.any(), (X[bad][:3], Z[bad][:3], got[bad][:3], want[bad][:3])
    # away from the boundaries nearly every quotient is settled
    k = int(np.ceil(np.log2(dim))) if dim > 1 else 0
    assert (~ok[half:]).mean() <= 2.5 * (2.0 ** (k - 25) + 2.0 ** -20) + 1e-4


def test_exact_halves_are_left_to_the_division():
    Z = F(np.array([1.0, 3.0, 1000.0, 0.125]))
    for base in (0.5, 7.5, 639.5, -0.5):
        _, ok = _settled(F(base) * Z, Z, 0, 1280)
        assert not ok.any()
