"""The exclusive scan behind the CSR partner lists and the flaw offsets where
its sums are large: past 2^30, up to 2^31 - 1 in 32-bit offsets, and past 2^32
in the 64-bit offsets of the partner lists."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def scan(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_03290_gb300 import build
    from paper_1604_03290_gb300 import sph
    sph.lib()
    so = str(tmp_path_factory.mktemp("scan") / "scan_check.so")
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-shared", os.path.join(ROOT, "tests", "native", "scan_check.cu"),
                    "-o", so, build.LIB, "-Xlinker", "-rpath=" + os.path.dirname(build.LIB), "-lcudart"],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(so)
    lib.scan_look_words.restype = ctypes.c_int64

    def run(counts, dtype):
        m = len(counts)
        x = torch.as_tensor(counts, dtype=torch.int32, device="cuda")
        out = torch.full((m,), -1, dtype=dtype, device="cuda")
        look = torch.full((lib.scan_look_words(ctypes.c_int64(m)),), -1, dtype=torch.int32, device="cuda")
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        f = lib.scan32 if dtype == torch.int32 else lib.scan64
        p = [ctypes.c_void_p(t.data_ptr()) for t in (x, out)]
        q = [ctypes.c_void_p(t.data_ptr()) for t in (look, err)]
        assert f(*p, ctypes.c_int64(m), *q, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        torch.cuda.synchronize()
        assert err.item() == 0
        return out.cpu().numpy()
    return run


@pytest.mark.parametrize("m", [1, 4096, 4097, 3 * 4096 + 5, 200 * 4096 + 1])
@pytest.mark.parametrize("total", [2 ** 20, 2 ** 30 - 1, 2 ** 30, 2 ** 30 + 2 ** 29, 2 ** 31 - 1])
def test_offsets_of_32_bits(scan, m, total):
    import torch
    rng = np.random.default_rng(m)
    cuts = np.sort(rng.integers(0, total + 1, m - 1)) if m > 1 else np.zeros(0, np.int64)
    counts = np.diff(np.concatenate([[0], cuts, [total]]))
    want = np.concatenate([[0], np.cumsum(counts)[:-1]])
    np.testing.assert_array_equal(scan(counts, torch.int32), want)


@pytest.mark.parametrize("m", [1, 4097, 3 * 4096 + 5, 200 * 4096 + 1])
def test_offsets_of_64_bits(scan, m):
    import torch
    counts = np.random.default_rng(m).integers(0, 2 ** 31, m)
    want = np.concatenate([[0], np.cumsum(counts)[:-1]])
    assert m == 1 or want[-1] > 2 ** 32
    np.testing.assert_array_equal(scan(counts, torch.int64), want)
