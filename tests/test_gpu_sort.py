"""The library's radix sort (GPU): results at the edges of its tiles, and a pass that
finds the sort failed moves nothing."""
import ctypes

import pytest

import paper_2009_12457_gb300 as bb

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

SORT_FAILED, GUARD = 8, 4096


def radix_sort(keys, alt, vals, vals_alt, count, bit_lo, bit_hi, err):
    """bbtc::radix_sort on the default stream; True when the result is in alt."""
    sort = bb.load()._ZN4bbtc10radix_sortEPmS0_PjS1_liiP11CUstream_stPiPb
    in_alt = ctypes.c_bool()
    ptr = [ctypes.c_void_p(t.data_ptr() if t is not None else None)
           for t in (keys, alt, vals, vals_alt)]
    torch.cuda.synchronize()
    assert sort(*ptr, ctypes.c_int64(count), bit_lo, bit_hi, None, ctypes.c_void_p(err.data_ptr()),
                ctypes.byref(in_alt)) == 0
    torch.cuda.synchronize()
    return in_alt.value


@pytest.mark.parametrize("with_vals", [False, True])
@pytest.mark.parametrize("count,bits", [(4095, 24), (4096, 17), (4097, 24), (100_000, 33),
                                        (100_000, 40)])
def test_sort(count, bits, with_vals):
    gen = torch.Generator("cuda").manual_seed(count + bits)
    keys = torch.randint(1 << bits, (count,), device="cuda", generator=gen)
    vals = torch.arange(count, dtype=torch.int32, device="cuda") if with_vals else None
    want, order = torch.sort(keys, stable=True)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    alt, vals_alt = torch.empty_like(keys), torch.empty_like(vals) if with_vals else None
    in_alt = radix_sort(keys, alt, vals, vals_alt, count, 0, bits, err)
    assert int(err) == 0
    assert torch.equal(alt if in_alt else keys, want)
    if with_vals:
        assert torch.equal((vals_alt if in_alt else vals).long(), order)


@pytest.mark.parametrize("with_vals", [False, True])
def test_passes_of_a_failed_sort_write_nothing(with_vals):
    count = 50_000
    keys = torch.randint(1 << 24, (count,), device="cuda")
    alt = torch.full((count + GUARD,), -1, dtype=torch.int64, device="cuda")
    vals = torch.arange(count, dtype=torch.int32, device="cuda") if with_vals else None
    vals_alt = torch.full((count + GUARD,), -1, dtype=torch.int32, device="cuda") if with_vals else None
    before = keys.clone()
    err = torch.full((1,), SORT_FAILED, dtype=torch.int32, device="cuda")
    radix_sort(keys, alt, vals, vals_alt, count, 0, 24, err)
    assert int(err) == SORT_FAILED
    assert torch.equal(keys, before) and bool((alt == -1).all())
    if with_vals:
        assert bool((vals_alt == -1).all()) and torch.equal(
            vals, torch.arange(count, dtype=torch.int32, device="cuda"))
