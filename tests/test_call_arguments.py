"""Arguments of the device calls as the native marshalling module takes them (no GPU: a host-only plan is refused by the library
after the arguments have been read)."""
import numpy as np
import pytest
import torch

import paper_2608_30386_b200 as dasc
from paper_2608_30386_b200 import binding


class Stream:
    cuda_stream = 0


T = torch.zeros(8)
IDX = torch.zeros(2, dtype=torch.int32)


@pytest.fixture(scope="module")
def plan():
    return dasc.dasc_plan(dasc.KDA, 1, 1, 1, 4, 4, np.zeros(4, np.float32), np.zeros(4, np.float32), w_max=16.0, device=-1)


def _copy(call, plan, layer_stride=16, req_stride=16, pool_arg=0):
    if "restore" in call.__name__:
        if "padded" in call.__name__:
            return call(plan, T, pool_arg, IDX, T, layer_stride, req_stride, IDX, stream=Stream())
        return call(plan, T, IDX, T, layer_stride, req_stride, IDX, pool_arg, stream=Stream())
    if "padded" in call.__name__:
        return call(plan, T, layer_stride, req_stride, IDX, T, pool_arg, IDX, stream=Stream())
    return call(plan, T, layer_stride, req_stride, IDX, T, IDX, pool_arg, stream=Stream())


def _refresh(plan, layer_stride=16, req_stride=16, total=1, longest=1, **kw):
    return dasc.dasc_refresh(plan, T, layer_stride, req_stride, IDX, T, T, T, T, T, IDX, total, longest, stream=Stream(), **kw)


def _window(plan, layer_stride=16, req_stride=16, total=1, window=1, **kw):
    return dasc.dasc_refresh_window(plan, T, layer_stride, req_stride, IDX, None, T, T, T, T, IDX, total, IDX, window=window,
                                    stream=Stream(), **kw)


def _reaches_the_library(call, *args, **kw):
    with pytest.raises(binding.DascError) as e:
        call(*args, **kw)
    assert e.value.status == binding.ERR_INVALID_ARG


COPIES = [dasc.dasc_pack, dasc.dasc_restore, dasc.dasc_pack_int8, dasc.dasc_restore_int8, dasc.dasc_pack_padded,
          dasc.dasc_restore_padded]


@pytest.mark.parametrize("call", COPIES, ids=lambda c: c.__name__)
def test_a_float_stride_of_a_copy_is_an_error(call, plan):
    _reaches_the_library(_copy, call, plan)
    _reaches_the_library(_copy, call, plan, layer_stride=np.int64(16), req_stride=np.int32(16))
    for name in ("layer_stride", "req_stride"):
        with pytest.raises(TypeError):
            _copy(call, plan, **{name: 16 / 2})
    if "padded" in call.__name__:
        _reaches_the_library(_copy, call, plan, pool_arg=4.0)   # a number of slots, taken by int()
    else:
        with pytest.raises(TypeError):
            _copy(call, plan, pool_arg=16 / 2)


@pytest.mark.parametrize("call", [_refresh, _window])
def test_whole_numbers_of_a_refresh(call, plan):
    _reaches_the_library(call, plan)
    for name in ("layer_stride", "req_stride", "layer_begin", "layer_end", "algo") + (("mode",) if call is _refresh else ()):
        with pytest.raises(TypeError):
            call(plan, **{name: 1.0})
    for name in ("total", "longest" if call is _refresh else "window"):
        _reaches_the_library(call, plan, **{name: 1.0})
        _reaches_the_library(call, plan, **{name: torch.tensor(1)})
    for scale in (1, 0.5, np.float32(0.5), torch.tensor(0.5)):
        _reaches_the_library(call, plan, q_scale=scale)
    with pytest.raises(TypeError):
        call(plan, q_scale=None)


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_the_current_stream_without_private_entries_of_torch(missing, monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_available", lambda: True)
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: type("S", (), {"cuda_stream": 77})())
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.setattr(torch._C, name, lambda *_: 1, raising=False)
    raw_stream, device = binding._stream_lookup()
    assert raw_stream(device()) == 1
    monkeypatch.delattr(torch._C, missing)
    raw_stream, device = binding._stream_lookup()
    assert raw_stream(device()) == 77
