"""Library calls from the binding's native module: what they take, what they refuse, and that the library sees the arguments as they are
(calls that end at the library's own checks or have nothing to do: no GPU is needed)."""
import ctypes

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
    (("x", 0, 0, 0, 4, 8, 1, 0, None, None, None, 0), AssertionError),                         # neither tensor, address nor None
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
