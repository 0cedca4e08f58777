"""Host-side checks of what the launches ask for, on the functions that the launch code itself calls (no GPU needed)."""
import ctypes as C
import functools

import pytest

from paper_2609_00355_b200 import binding
from paper_2609_00355_b200 import build as glance_build

SM_SMEM, PER_CTA, SM_COLUMNS = 228 * 1024, 1024, 512      # shared memory of an SM, the share each CTA loses, tensor memory


class CtaSize(C.Structure):
    _fields_ = [("smem", C.c_longlong), ("columns", C.c_longlong)]


@pytest.fixture(scope="module")
def lib():
    glance_build.build()
    return binding.load_library()


def _attention_sizes(lib):
    fn = lib._ZN6glance21attention_tc_cta_sizeEi
    fn.restype, fn.argtypes = CtaSize, [C.c_int]
    return [fn(d) for d in (64, 128)]


def _gemm_sizes(lib):
    tc = lib._ZN6glance11tc_cta_sizeEiiiib
    tc.restype, tc.argtypes = CtaSize, [C.c_int] * 4 + [C.c_bool]
    wide = lib._ZN6glance13wide_cta_sizeEiiiib
    wide.restype, wide.argtypes = CtaSize, [C.c_int] * 4 + [C.c_bool]
    out = []
    for R in list(range(1, 129)) + [129, 144, 160, 161, 257, 577, 1280]:
        for mode, two in ((0, False), (1, True), (1, False), (2, False), (3, True), (4, False), (5, False)):
            for Nout in (256, 4608, 37888, 152064):
                for S in (1, 2, 8) if mode in (3, 4) else (1,):
                    out.append(tc(mode, Nout, R, S, two))
        if R > 128:
            out += [wide(mode, 8192, 4096, R, mode in (1, 3)) for mode in (1, 2, 3, 4)]
    return out


def _most_columns(sizes):
    """The most columns that CTAs which fit an SM's shared memory together can want."""
    items = sorted({(s.smem + PER_CTA, s.columns) for s in sizes})

    @functools.lru_cache(maxsize=None)
    def most(room):
        return max([c + most((room - b) // 64 * 64) for b, c in items if b <= room], default=0)

    return most(SM_SMEM)


def test_ctas_that_fit_an_sm_fit_its_tensor_memory(lib):
    """A CTA that waits for columns, held by one that waits for it, would wait for good: shared memory alone has to keep such
    CTAs apart (the kernels' register counts do not count here)."""
    sizes = _attention_sizes(lib) + _gemm_sizes(lib)
    assert all(0 < s.smem <= 227 * 1024 and s.columns <= SM_COLUMNS for s in sizes)
    assert _most_columns(sizes) <= SM_COLUMNS
