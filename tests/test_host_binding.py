"""The binding's native step calls without a GPU: what they accept as tensors and streams, what they refuse, return codes."""
import pytest
import torch

from paper_2511_16047_b200 import binding as B


class _Stream:
    cuda_stream = 0


def _plan(layers=1, sides=(1, 2, 3), flags=B.FLAG_PLAN_ONLY):
    desc, keep = B.make_desc(layers, 2, 64, 2, sides, [(1, 1, True)] * layers, flags=flags)
    return B.amskv_cache_create(desc)


def _views(t):
    x = torch.zeros(2, t, 3, 2, 64, dtype=torch.bfloat16)
    return [x[:, :, i].transpose(1, 2) for i in range(3)]


def test_tensors_addresses_and_none_are_accepted():
    c = _plan()
    q, k, v = _views(1)
    B.amskv_append_attend(c, 0, 0, k, v, q, q, _Stream())              # strided views
    k4 = torch.zeros(2, 2, 4, 64, dtype=torch.bfloat16)
    B.amskv_append(c, 0, 1, k4, k4.data_ptr(), stream=0)               # a contiguous tensor beside a raw address
    B.amskv_append(cache=c, layer=0, scale=2, K=None, V=None)          # bookkeeping only
    assert B.amskv_kept_segments(c, 0, 2) == [0, 1, 2]
    B.amskv_cache_destroy(c)


def test_mismatched_and_malformed_tensors_are_refused():
    c = _plan(sides=(2, 2))
    q, k, v = _views(4)
    with pytest.raises(ValueError):
        B.amskv_append(c, 0, 0, k, v.contiguous())                     # one strided, one contiguous
    with pytest.raises(ValueError):
        B.amskv_append_attend(c, 0, 0, k, v[:1].expand(2, 2, 4, 64), q, q)
    with pytest.raises(AssertionError):
        B.amskv_append(c, 0, 0, k.transpose(2, 3), v.transpose(2, 3))  # channels not contiguous
    with pytest.raises(TypeError):
        B.amskv_append(c, 0, 0, object(), object())
    assert B.amskv_kept_segments(c, 0, 0) == [0]
    with pytest.raises(B.AmskvError) as e:
        B.amskv_append(c, 0, 1, k, v)                                  # nothing above went through: scale 0 is still next
    assert e.value.code == B.ERR_ORDER
    with pytest.raises(B.AmskvError) as e:
        B.amskv_attend(c, 0, 0, q, q)
    assert e.value.code == B.ERR_UNSUPPORTED
    with pytest.raises(B.AmskvError) as e:
        B.amskv_append(None, 0, 0, k, v)
    assert e.value.code == B.ERR_INVALID
    with pytest.raises(OverflowError):
        B.amskv_append(c, 1 << 40, 0, k, v)
    B.amskv_cache_destroy(c)


@pytest.mark.parametrize("native", [True, False], ids=["native", "ctypes"])
def test_what_ctypes_takes_the_step_calls_take(native, monkeypatch):
    """The native module serves the usual forms of arguments and leaves every other to ctypes: a handle object is accepted,
    what ctypes refuses is refused, and without the module everything goes through ctypes."""
    import ctypes
    if not native:
        monkeypatch.setattr(B, "_steps", None)
    c = _plan(layers=2, sides=(1, 2))
    q, k, v = _views(1)
    B.amskv_append(ctypes.c_void_p(c), 0, 0, k, v)
    B.amskv_append_attend(ctypes.c_void_p(c), 1, 0, k, v, q, q)
    B.amskv_append(c, ctypes.c_int(0), True, k.data_ptr(), ctypes.c_void_p(k.data_ptr()).value)
    assert B.amskv_kept_segments(c, 0, 1) == [0, 1]
    for bad in (float(c), torch.tensor(1)):
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            B.amskv_append(bad, 1, 1, k, v)
    for bad in (1.0, "1"):
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            B.amskv_append(c, 1, bad, k, v)
    with pytest.raises(ValueError):
        B.amskv_append(c, 1, 1, k, v.contiguous())
    with pytest.raises(AssertionError):
        B.amskv_attend(c, 1, 0, q.transpose(2, 3), q)
    with pytest.raises(OverflowError):
        B.amskv_attend(c, 0, 1 << 31, q, q)
    B.amskv_append(c, 1, 1, k, v)                                      # none of them went through
    B.amskv_cache_destroy(c)
