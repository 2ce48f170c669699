"""The CPython entry points: how arguments become pointers and numbers, and how a status becomes an exception (no GPU:
the calls below are refused by the library's own checks before any CUDA call)."""
import ctypes

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


@pytest.mark.parametrize("make", [lambda: np.int64(4096), lambda: np.float32(1.0), lambda: np.bool_(True), lambda: b"0123456789abcdef",
                                  lambda: bytearray(64), lambda: memoryview(bytearray(64)), lambda: ctypes.create_string_buffer(64)],
                         ids=["numpy integer", "numpy float", "numpy bool", "bytes", "bytearray", "memoryview", "ctypes array"])
def test_objects_with_storage_of_their_own_are_not_pointers(make):
    """The address of a scalar's or a byte string's storage is not an array: T = 0 keeps the library from using it."""
    with pytest.raises(AttributeError):
        scan(make(), T=0)


def test_contexts_are_integers_and_scalars_are_converted_as_python_does():
    args = (None, None, None, 0, 0, 0, None, None, None, None, None, 0)   # a null frame pointer: refused before the context is used
    for ctx in (np.zeros(4), np.int64(4096), b"x", 1.5):
        with pytest.raises(ctypes.ArgumentError):
            hts.hts_policy_step(ctx, *args)
    for ctx in (None, 4096, ctypes.c_void_p(), ctypes.c_void_p(4096)):
        with pytest.raises(hts.HtsError) as e:
            hts.hts_policy_step(ctx, *args)
        assert e.value.status == 1
    with pytest.raises(hts.HtsError):
        scan(np.zeros((2, 3), np.float32), gamma="0.5", lam=np.float32(0.5), T="0")
    with pytest.raises(ValueError):
        scan(np.zeros((2, 3), np.float32), gamma="half")
