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


RESIDENT = {1: 148, 2: 74, 3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15}     # clusters of a size at one CTA per SM


@pytest.mark.parametrize("two_term", [False, True])
def test_launches_with_a_whole_sm_to_a_cta_are_resident_at_once(lib, two_term):
    """A ring that takes an SM for itself must not leave clusters of the launch to a second wave, and the planes of a cluster's
    splits fit the ring."""
    splits = lib._ZN6glance9tc_splitsEiiib
    splits.restype, splits.argtypes = C.c_int, [C.c_int] * 3 + [C.c_bool]
    size = lib._ZN6glance11tc_cta_sizeEiiiib
    size.restype, size.argtypes = CtaSize, [C.c_int] * 4 + [C.c_bool]
    for tiles in range(1, 80):
        for ktiles in (1, 2, 8, 20, 36, 96, 296):
            for R in (1, 16, 32, 65, 96, 128, 132, 192, 320, 600, 1100):
                S = splits(128 * tiles, 64 * ktiles, R, two_term)
                blocks = -(-R // 128)
                rows = -(-(-(-R // blocks)) // 16) * 16
                s = size(3 if two_term else 4, 128 * tiles, R, S, two_term)
                assert 1 <= S <= min(8, ktiles)
                assert S * -(-rows // S) * 512 <= s.smem - 1024
                if 2 * (s.smem + PER_CTA) > SM_SMEM:
                    assert tiles * blocks <= RESIDENT[S], (tiles, ktiles, R, S)


@pytest.mark.parametrize("hidden,K,rows,S", [(2816, 7680, 384, 4), (1792, 4864, 768, 3), (2816, 2816, 512, 3), (3328, 8960, 256, 5),
                                             (3584, 3584, 144, 4), (2304, 2304, 1280, 1)])
def test_split_factors_use_the_clusters_that_fit_at_two_ctas_an_sm(lib, hidden, K, rows, S):
    """66 clusters of four and 84 of three are one wave; 180 of three would be two full ones for an unsplit one."""
    splits = lib._ZN6glance9tc_splitsEiiib
    splits.restype, splits.argtypes = C.c_int, [C.c_int] * 3 + [C.c_bool]
    assert splits(hidden, K, rows, True) == S


@pytest.mark.parametrize("rows,spans,warps,k,resident,one", [
    (15, 149, 19, 1, 15, True), (16, 149, 19, 1, 15, False), (45, 149, 19, 8, 15, True), (60, 149, 19, 4, 15, False),
    (98, 149, 19, 8, 15, False), (142, 9, 2, 1, 142, True), (143, 9, 2, 16, 142, False), (90, 64, 8, 4, 48, False),
    (80, 64, 8, 4, 48, True), (16, 98, 13, 16, 15, False), (480, 8, 8, 4, 444, True), (3000, 8, 8, 16, 444, False)])
def test_topk_takes_one_launch_while_its_clusters_are_resident(lib, rows, spans, warps, k, resident, one):
    fn = lib._ZN6glance15topk_one_launchEiiiii
    fn.restype, fn.argtypes = C.c_bool, [C.c_int] * 5
    assert fn(rows, spans, warps, k, resident) is one
