"""Library calls from the binding's native module: what they take, what they refuse, and that the library sees the arguments as they are
(calls that end at the library's own checks or have nothing to do: no GPU is needed)."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2603_20586_b200 as mka
from paper_2603_20586_b200 import binding as b

H = b._host_args


def _shape(**kw):
    return mka.make_shape(**{**dict(B=1, H=2, T=8, d=64, D=64, window=4), **kw})


def test_status_is_the_librarys():
    X, W, g = torch.zeros(4, 8), torch.zeros(8, 3), torch.zeros(4, 3)
    assert H.call_router(b._router, X, W, None, 0, 8, 1, 0, g, None, None, 0) == 0            # no rows
    assert H.call_router(b._router, X, W, None, 4, 0, 1, 0, g, None, None, 0) == 2            # D = 0
    assert H.call_router(b._router, X, W, None, 4, 8, 7, 0, g, None, None, 0) == 1            # no such dtype
    assert H.call_router(b._router, None, W, None, 4, 8, 1, 0, g, None, None, 0) == 1         # no rows given
    none = [None] * 3
    lv, gr = b._levels(none, none), H.grads(none, none, none)
    pl = b._paged_levels(none, none, none, None, (0, 0, 0))
    empty, bad = _shape(T=0), _shape(d=48)
    assert H.call_fwd(b._fwd, empty, None, lv, None, None, None, None, 0, None, 0, 0) == 0
    assert H.call_fwd(b._fwd, bad, None, lv, None, None, None, None, 0, None, 0, 0) == 2
    assert H.call_fwd_paged(b._fwd_paged, empty, 1, None, pl, None, None, None, None, 0, None, 0, 0) == 0
    assert H.call_fwd_paged(b._fwd_paged, empty, 3, None, pl, None, None, None, None, 0, None, 0, 0) == 2      # 2 heads on 3
    assert H.call_decode(b._decode, _shape(T=8), None, lv, None, None, None, None, 0, 0) == 2                  # T != 1
    assert H.call_decode_paged(b._decode_paged, _shape(T=1), 1, None, pl, None, None, None, None, 0, 0) == 1   # no queries
    assert H.call_bwd(b._bwd, bad, None, lv, None, None, None, None, None, 0, None, gr, None, None, None, None, 0, 0) == 2


@pytest.mark.parametrize("args,error", [
    ((1,), AssertionError),                                                                    # too few
    (("x", 0, 0, 0, 4, 8, 1, 0, None, None, None, 0), AssertionError),                         # neither tensor nor None
    ((None, None, None, 4.0, 8, 1, 0, None, None, None, 0), TypeError),                        # a float for a count
    ((None, None, None, 2 ** 70, 8, 1, 0, None, None, None, 0), OverflowError),
])
def test_router_arguments_that_are_refused(args, error):
    with pytest.raises(error):
        H.call_router(b._router, *args)


@pytest.mark.parametrize("shape,levels,error", [
    (b"short", None, TypeError), (None, None, TypeError), ("ok", b"\0" * 143, AssertionError), ("ok", None, AssertionError)])
def test_shapes_and_levels_that_are_refused(shape, levels, error):
    lv = b._levels([None] * 3, [None] * 3)
    assert len(lv) == 3 * ctypes.sizeof(b.mka_level)
    with pytest.raises(error):
        H.call_decode(b._decode, _shape(T=1) if shape == "ok" else shape, None, lv if levels is None and shape != "ok" else levels, None, None, None,
                      None, 0, 0)


def test_row_counts():
    K = [torch.zeros(1, 1, 5, 4), None, torch.zeros(1, 1, 0, 4)]
    assert b._row_counts(K) == (5, 0, 0) == b._row_counts(tuple(K)) == b._row_counts(dict(enumerate(K)))


class _Legacy:
    cuda_stream = 0                                           # (asking for the current stream would need a GPU)


def _calls():
    """Each call of the public functions with nothing to launch, and the names of its arguments that are memory."""
    none, n = [None] * 3, dict(stream=_Legacy())
    Q, q = torch.zeros(1, 2, 0, 64, dtype=torch.bfloat16), torch.zeros(0, 2, 64, dtype=torch.bfloat16)
    g, lse, ws, X, W = torch.zeros(1, 0, 3), torch.zeros(1, 2, 0), torch.zeros(256, dtype=torch.uint8), torch.zeros(0, 8), torch.zeros(8, 3)
    seqs, steps = _shape(T=0), _shape(B=0, T=1)
    out = dict(O=torch.zeros(1, 2, 0, 64), LSE=lse)
    return {
        "router": (mka.mka_router, dict(R=X, W_r=W, b_r=None, gate=g, **n), ("b_r", "gate", "log2_gate", "route_idx")),
        "fwd": (mka.mka_fwd, dict(shape=seqs, Q=Q, K=none, V=none, gate=g, ws=ws, **out, **n), ("Q", "gate", "O", "LSE", "ws")),
        "fwd_paged": (mka.mka_fwd_paged, dict(shape=seqs, H_kv=2, Q=Q, pools_k=none, pools_v=none, tables=none, n=(0, 0, 0), gate=g, ws=ws, **out, **n),
                      ("Q", "gate", "O", "LSE", "ws")),
        "decode": (mka.mka_decode, dict(shape=steps, q=q, K=none, V=none, gate=g, ws=ws, **out, **n), ("q", "gate", "O", "LSE", "ws")),
        "decode_paged": (mka.mka_decode_paged, dict(shape=steps, H_kv=2, q=q, pools_k=none, pools_v=none, tables=none, n=(0, 0, 0), gate=g, ws=ws, **out, **n),
                         ("q", "gate", "O", "LSE", "ws")),
        "bwd": (mka.mka_bwd, dict(shape=seqs, Q=Q, K=none, V=none, gate=g, O=Q, LSE=lse, dO=Q, ws=ws, **n),
                ("Q", "gate", "O", "LSE", "dO", "R", "dQ", "dG", "dW_r", "db_r", "ws")),
    }


@pytest.mark.parametrize("name", ["router", "fwd", "fwd_paged", "decode", "decode_paged", "bwd"])
def test_numbers_are_no_memory(name):
    function, args, memory = _calls()[name]
    function(**args)
    for key in memory:
        for wrong in (True, False, 0, 1, 2 ** 40):
            with pytest.raises((AssertionError, AttributeError)):
                function(**{**args, key: wrong})


def test_every_pointer_of_a_native_call_refuses_numbers():
    none = [None] * 3
    lv, gr, pl = b._levels(none, none), H.grads(none, none, none), b._paged_levels(none, none, none, None, (0, 0, 0))
    empty, step = _shape(T=0), _shape(B=0, T=1)
    for call, address, args in [
            (H.call_router, b._router, (None, None, None, 0, 8, 1, 0, None, None, None)),
            (H.call_fwd, b._fwd, (empty, None, lv, None, None, None, None, 0, None, 0)),
            (H.call_fwd_paged, b._fwd_paged, (empty, 1, None, pl, None, None, None, None, 0, None, 0)),
            (H.call_decode, b._decode, (step, None, lv, None, None, None, None, 0)),
            (H.call_decode_paged, b._decode_paged, (step, 1, None, pl, None, None, None, None, 0)),
            (H.call_bwd, b._bwd, (empty, None, lv, None, None, None, None, None, 0, None, gr, None, None, None, None, 0))]:
        for i, x in enumerate(args):
            if x is not None:
                continue
            for wrong in (True, 0, 8):
                with pytest.raises(AssertionError):
                    call(address, *args[:i], wrong, *args[i + 1:], 0)
        for wrong in (1.0, torch.zeros(1)):                    # nor is a tensor a stream
            with pytest.raises(AssertionError):
                call(address, *args, wrong)


@pytest.mark.parametrize("whole", [np.int64, np.int32, torch.tensor, int])
def test_counts_may_be_whole_numbers_of_any_kind(whole):
    calls = _calls()
    for name, key, value in (("router", "route", 1), ("fwd_paged", "H_kv", 2), ("decode_paged", "H_kv", 2)):
        function, args, _ = calls[name]
        function(**{**args, key: whole(value)})
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            function(**{**args, key: float(value)})


def test_memory_and_streams_of_other_kinds():
    function, args, _ = _calls()["router"]
    function(**{**args, "log2_gate": torch.zeros(4).untyped_storage()})
    for handle in (ctypes.c_void_p(0), ctypes.c_void_p(), None):
        stream = _Legacy()
        stream.cuda_stream = handle
        function(**{**args, "stream": stream})


@pytest.mark.parametrize("name", ["fwd", "fwd_paged", "decode", "decode_paged", "bwd"])
def test_only_a_shape_is_a_shape(name):
    native = {"fwd": (H.call_fwd, b._fwd), "fwd_paged": (H.call_fwd_paged, b._fwd_paged), "decode": (H.call_decode, b._decode),
              "decode_paged": (H.call_decode_paged, b._decode_paged), "bwd": (H.call_bwd, b._bwd)}[name]
    none = [None] * 3
    lv, gr, pl = b._levels(none, none), H.grads(none, none, none), b._paged_levels(none, none, none, None, (0, 0, 0))
    rest = {"fwd": (None, lv, None, None, None, None, 0, None, 0, 0), "fwd_paged": (1, None, pl, None, None, None, None, 0, None, 0, 0),
            "decode": (None, lv, None, None, None, None, 0, 0), "decode_paged": (1, None, pl, None, None, None, None, 0, 0),
            "bwd": (None, lv, None, None, None, None, None, 0, None, gr, None, None, None, None, 0, 0)}[name]
    shape = _calls()[name][1]["shape"]

    class Own(mka.mka_shape):
        pass

    native[0](native[1], Own.from_buffer_copy(shape), *rest)
    for wrong in (bytes(shape), bytearray(shape), np.frombuffer(bytes(shape), dtype=np.uint8), (ctypes.c_int32 * 12).from_buffer_copy(shape)):
        with pytest.raises(TypeError):
            native[0](native[1], wrong, *rest)


@pytest.mark.parametrize("args,message", [
    ((1,), "number of arguments"),
    ((None, "x", None, 0, 8, 1, 0, None, None, None, 0), "a tensor"),
    ((None, None, None, 0, 8, 1, 0, None, True, None, 0), "a tensor"),
    ((None, None, None, 0, 8, 1, 0, None, None, None, 1.0), "an address"),
])
def test_refusals_say_what_is_wrong(args, message):
    with pytest.raises(AssertionError, match=message):
        H.call_router(b._router, *args)
    with pytest.raises(AssertionError, match="the address of a function"):
        H.call_router(0, None, None, None, 0, 8, 1, 0, None, None, None, 0)
    with pytest.raises(AssertionError, match="levels"):
        H.call_decode(b._decode, _shape(T=1), None, b"", None, None, None, None, 0, 0)
