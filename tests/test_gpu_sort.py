"""The stable radix sort against numpy's: both forms of a pass (few keys, many),
partial tiles, one to seven digits, equal keys; and with a poll limit of zero,
where a tile counts the keys before it instead of waiting for their counts."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# tiles hold 1024 .. 8192 keys; many keys: from about 1.2 million
SIZES = [1, 2, 31, 1023, 1024, 1025, 16385, 70001, 311297, 1244000, 1246000, 2500001]


def _sort(key, bits, spins):
    from paper_1706_06989_gb300 import fmm
    s = fmm.FMM()
    f = s.lib.fmm_debug_sort
    f.restype = ctypes.c_int
    f.argtypes = [ctypes.c_void_p, ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int64] + [ctypes.c_int] * 2 + [
        ctypes.c_void_p] * 2
    k = torch.from_numpy(key.view(np.int64 if key.itemsize == 8 else np.int32)).cuda()
    v = torch.arange(len(key), dtype=torch.int32, device="cuda")
    ok, ov = torch.empty_like(k), torch.empty_like(v)
    torch.cuda.synchronize()
    rc = f(s._h, key.itemsize, k.data_ptr(), v.data_ptr(), len(key), bits, spins, ok.data_ptr(), ov.data_ptr())
    assert rc == fmm.FMM_OK
    return ok.cpu().numpy().view(key.dtype), ov.cpu().numpy()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("dtype,bits", [(np.uint32, 1), (np.uint32, 10), (np.uint32, 14), (np.uint32, 20),
                                        (np.uint32, 31), (np.uint64, 9), (np.uint64, 63)])
def test_sort(n, dtype, bits):
    rng = np.random.default_rng(n + bits)
    key = rng.integers(0, 1 << bits, n, dtype=dtype)
    key[: n // 3] = key[0]  # many equal keys
    order = np.argsort(key, kind="stable")
    for spins in (1 << 16, 0):
        if spins == 0 and n > 400000:
            continue
        k, v = _sort(key, bits, spins)
        assert np.array_equal(k, key[order]) and np.array_equal(v, order)
