"""The FP64 reciprocals of csrc/fp64fast.cuh to the error their derivation gives,
in units in the last place of the result (ulp).  With a seed of 20 bits, e is
below 2^-20 (1/x) or 2^-19 (1/sqrt(x)) and what the step leaves out below e^3
2^53 = 0.008 and (5/16) e^3 2^53 = 0.02 ulp.  1/x: one last rounding, 0.5 ulp.
1/sqrt(x): also the rounding of x y, 2^-53, which enters halved (at most 0.5
ulp, at mantissas just below 2): 1.0 in all.  Two correctly rounded operations,
1 / sqrt(x), reach 1.5."""
import numpy as np
import pytest

from test_gpu_fp64_forms import forms  # noqa: F401  (the fixture that runs both on the device)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(0, 0), (-40, 40), (-958, 959)])
def test_within_the_derived_error(forms, lo, hi):  # noqa: F811
    rng = np.random.default_rng(hi + 5)
    x = rng.uniform(1.0, 2.0, 1 << 21)
    x[:4] = 1.0, np.nextafter(1.0, 2.0), 2.0, np.nextafter(2.0, 1.0)
    x = np.ldexp(x, rng.integers(lo, hi + 1, len(x)))
    rcp, rsq = forms(x)
    xl = x.astype(np.longdouble)
    for got, want, bound in ((rcp, 1 / xl, 0.51), (rsq, 1 / np.sqrt(xl), 1.02)):
        ulp = np.spacing(want.astype(np.float64)).astype(np.longdouble)
        assert (np.abs(got.astype(np.longdouble) - want) / ulp).max() <= bound
