"""FP64 trial spins carry their last digits at every size of a component, near
the poles and the axes too, on all of its launches' shared form: a sweep at
beta = 0 leaves every site at its trial; the smallest components of two million
sites, and others at random, against decimal arithmetic on the same uniforms.

Bound in units of the last place: the sine of a table step is off by at most 4
units of 2^-63, and is 2^-10.4 at least where it does not come from the angle
itself; the product with r, a mantissa of 1/4 or more, drops at most 3 units of
2^-61 of it: 4 2^-52.6 + 3 2^-50.6 of the component, 22 units, and one for the
last rounding.
"""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_2106_11286_gb300 import hs

pytestmark = pytest.mark.gpu

getcontext().prec = 60
PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494459")
ONE = 1 << 52


def _sin(x):
    term = total = x
    for k in range(1, 40):
        term *= -x * x / ((2 * k) * (2 * k + 1))
        total += term
    return total


def _cos(x):
    term = total = Decimal(1)
    for k in range(1, 40):
        term *= -x * x / ((2 * k - 1) * (2 * k))
        total += term
    return total


def _sphere_point(iz, iv):
    z = Decimal(iz - ONE) / ONE
    r = ((1 - z) * (1 + z)).sqrt()
    quarter, f = divmod(iv, 1 << 51)  # pi t = (quarter + f 2^-51) pi / 2
    if f <= 1 << 50:
        a = PI / 2 * f / (1 << 51)
        s, c = _sin(a), _cos(a)
    else:
        a = PI / 2 * ((1 << 51) - f) / (1 << 51)
        s, c = _cos(a), _sin(a)
    s, c = ((s, c), (c, -s), (-s, -c), (-c, s))[quarter]
    return -r * c, -r * s, z


@pytest.mark.parametrize("kind,dims", [("sc", (128, 128, 128)), ("sc", (96, 96, 96)), ("bcc", (64, 64, 64))])
def test_trial_components_to_their_last_digits(orc, kind, dims):
    with hs.Lattice(kind, dims=dims, precision="fp64", seed=29) as lat:
        lat.init()
        lat.set_sweep_counter(6)
        lat.sweep(0.0, 1)
        S = lat.get_spins()
        assert lat.measure()["accept_rate"] == 1.0
    colour = orc.colour_structured(kind, dims)
    small = np.argsort(np.abs(S[:, :2]).min(1))[:400]
    rest = np.random.default_rng(1).integers(0, len(S), 200)
    assert np.abs(S[small, :2]).min() < 2.0**-18
    for i in np.concatenate((small, rest)):
        uz, uv, _ = orc.trial_uniforms(0, seed=29, replica=0, site=int(i), rank=0, sweep_index=6, colour=int(colour[i]))
        want = _sphere_point(int(uz * 2.0**53), int(uv * 2.0**53))
        for q in range(3):
            off = abs(Decimal(float(S[i, q])) - want[q])
            assert off <= 23 * Decimal(float(np.spacing(abs(S[i, q])))), (i, q, S[i, q], want[q])
