"""The FP64 reciprocal and reciprocal square root of the FP64 pair loops
(csrc/fp64fast.cuh) against correctly rounded references: within two units in
the last place over their fast range, exactly the language's operations outside
it (zero, subnormals, both ends of the exponent range, infinities, NaN).  And
the FP64 right-hand side against the oracle at sizes whose partner lists are
shared by 8, 4, 2 and 1 lanes (rhs_passes)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl
from parity_util import check_damage, compare_rhs, flawed

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_03290_gb300 import build
    so = str(tmp_path_factory.mktemp("fp64") / "fp64fast_check.so")
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-shared", os.path.join(ROOT, "tests", "native", "fp64fast_check.cu"),
                    "-o", so, "-lcudart"], check=True, capture_output=True)
    lib = ctypes.CDLL(so)

    def run(x):
        t = torch.as_tensor(x, dtype=torch.float64, device="cuda")
        a, b = torch.empty_like(t), torch.empty_like(t)
        assert lib.fp64_forms(ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(a.data_ptr()),
                              ctypes.c_void_p(b.data_ptr()), t.numel(),
                              ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        torch.cuda.synchronize()
        return a.cpu().numpy(), b.cpu().numpy()
    return run


@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (-60.0, 60.0), (-959.0, 961.0)])
def test_within_two_ulps(forms, lo, hi):
    rng = np.random.default_rng(3)
    x = np.exp2(rng.uniform(lo, hi, 1 << 20)) * rng.uniform(1.0, 2.0, 1 << 20)
    rcp, rsq = forms(x)
    xl = x.astype(np.longdouble)
    for got, want in ((rcp, 1 / xl), (rsq, 1 / np.sqrt(xl))):
        ulp = np.spacing(want.astype(np.float64)).astype(np.longdouble)
        assert (np.abs(got.astype(np.longdouble) - want) / ulp).max() <= 2.0


def test_outside_the_fast_range(forms):
    x = np.array([0.0, 5e-324, 1e-310, 2.0 ** -1022, 2.0 ** -960, 2.0 ** 962, 1.7e308, np.inf])
    rcp, rsq = forms(x)
    with np.errstate(divide="ignore", over="ignore"):
        np.testing.assert_array_equal(rcp, 1.0 / x)
        want = 1.0 / np.sqrt(x)
    want[0] = 0.0  # coincident particles: no direction
    np.testing.assert_array_equal(rsq, want)
    rcp, rsq = forms(np.array([np.nan, -2.0]))
    assert np.isnan(rcp[0]) and rcp[1] == -0.5 and not rsq.any()


@pytest.mark.parametrize("n_side", [6, 13, 20, 24, 28])
def test_rhs_with_shared_lists(n_side):
    import oracle
    from paper_1604_03290_gb300 import sph
    ps = flawed(wl.measurement_1m(seed=17, n_side=n_side))
    o = oracle.rhs(ps, ps.materials, ps.params)
    out = sph.rhs(sph.Context(3, ps.n, max_neighbours=160), sph.DeviceState(ps), ps.materials, ps.params)
    g = {k: v.cpu().numpy() for k, v in out.items()}
    np.testing.assert_array_equal(g["nnb"], o["nnb"])
    compare_rhs(ps, o, g, 1e-12)  # the tolerance of the FP64 parity tests
    check_damage(ps, o, g, "fp64", 1e-12)
