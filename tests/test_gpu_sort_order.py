"""The sample sort's permutation itself, against numpy's stable argsort of the keys: one block up to
4096 keys of at most 20 bits, radix passes over 2048-key tiles above, one pass and two, few and many
equal keys, keys at the ends of their range; and the 64-bit sort of the same passes."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class SkyGrid(C.Structure):   # of which the sort reads n_cells
    _fields_ = [("order", C.c_int), ("n_cells", C.c_int), ("mode", C.c_int), ("gmst", C.c_double),
                ("x", C.c_double * 9), ("span", C.c_double * 3)]


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_11655_gb300 as G
    L = G.load(build_if_missing=True)
    out = {}
    p = C.c_void_p
    for name, sym, res, args in (
            ("words", "_ZN4rift18sort_scratch_wordsEl", C.c_size_t, [C.c_int64]),
            ("words64", "_ZN4rift20sort64_scratch_wordsEl", C.c_size_t, [C.c_int64]),
            ("sort", "_ZN4rift11launch_sortERKNS_7SkyGridEPKjlPjS5_P11CUstream_stPi", C.c_int,
             [C.POINTER(SkyGrid), p, C.c_int64, p, p, p, p]),
            ("sort64", "_ZN4rift13launch_sort64EPmS0_liPjP11CUstream_stPi", C.c_int,
             [p, p, C.c_int64, C.c_int, p, p, p])):
        f = getattr(L, sym)
        f.restype, f.argtypes = res, args
        out[name] = f
    return out


COUNTS = [1, 2, 31, 1000, 2048, 4095, 4096, 4097, 6143, 6145, 300001]


@pytest.mark.parametrize("cells", [1, 16, 1000, 1024, 6 << 12, 6 << 16, 1 << 20])
def test_order_and_stability(lib, cells):
    import torch
    rng = np.random.default_rng(cells)
    for n in COUNTS:
        for keys in (rng.integers(0, cells, n), rng.integers(0, min(cells, 5), n), np.full(n, cells - 1),
                     np.arange(n)[::-1] % cells):
            k = torch.from_numpy(keys.astype(np.uint32).view(np.int32)).cuda()
            scratch = torch.empty(lib["words"](n), dtype=torch.int32, device="cuda")
            perm = torch.full((n,), -1, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            grid = SkyGrid(n_cells=cells)
            assert lib["sort"](C.byref(grid), k.data_ptr(), n, scratch.data_ptr(), perm.data_ptr(), None, None) == 0
            torch.cuda.synchronize()
            assert np.array_equal(perm.cpu().numpy(), np.argsort(keys, kind="stable"))


@pytest.mark.parametrize("bits", [1, 10, 11, 37, 63])
def test_64_bit_keys(lib, bits):
    import torch
    rng = np.random.default_rng(bits)
    for n in COUNTS:
        keys = rng.integers(0, 1 << bits, n)
        k = torch.from_numpy(keys.copy()).cuda()
        tmp = torch.empty_like(k)
        scratch = torch.empty(lib["words64"](n), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib["sort64"](k.data_ptr(), tmp.data_ptr(), n, bits, scratch.data_ptr(), None, None) == 0
        torch.cuda.synchronize()
        assert np.array_equal(k.cpu().numpy(), np.sort(keys))
