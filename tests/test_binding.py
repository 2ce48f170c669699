"""The CPython entry points: how arguments become pointers and numbers, and how a status becomes an exception (no GPU:
the calls below are refused by the library's own checks before any CUDA call)."""
import numpy as np
import pytest

import paper_2012_09849_b200 as hts

SCAN = dict(gamma=0.99, lam=0.95, T=2, N=3)


def scan(r, stream=0, **kw):
    a = np.zeros((2, 3), np.float32)
    k = {**SCAN, **kw}
    return hts.hts_gae(r, a, np.zeros((2, 3), np.uint8), np.zeros(3, np.float32), k["gamma"], k["lam"], k["T"], k["N"], a.copy(), a.copy(), stream)


@pytest.mark.parametrize("kw", [dict(T=0), dict(N=np.int64(0)), dict(gamma=float("nan")), dict(lam=2), dict(T=True, N=-1)])
def test_refusals_carry_the_status_and_the_name(kw):
    with pytest.raises(hts.HtsError) as e:
        scan(np.zeros((2, 3), np.float32), **kw)
    assert e.value.status == 1 and "hts_gae: HTS_ERR_INVALID_ARG" in str(e.value)


def test_pointers_may_be_none_integers_arrays_or_have_a_stream_attribute():
    class Stream:
        cuda_stream = 0
    for r in (None, 0):                                   # a null pointer is refused by the library, not by the binding
        with pytest.raises(hts.HtsError) as e:
            scan(r, stream=Stream())
        assert e.value.status == 1
    with pytest.raises(AssertionError):
        scan(np.zeros((4, 3), np.float32)[::2])
    with pytest.raises(AttributeError):
        scan(object())
    with pytest.raises(ValueError):                       # int("two")
        scan(np.zeros((2, 3), np.float32), T="two")


def test_weights_are_taken_by_name():
    with pytest.raises(KeyError):
        hts.hts_policy_load_weights(0, {}, 0)
    with pytest.raises(hts.HtsError) as e:
        hts.hts_policy_load_weights(0, {k: 0 for k in hts.WEIGHT_NAMES}, 0)
    assert e.value.status == 1 and "hts_policy_load_weights" in str(e.value)
