"""The binding's native marshalling: the words it writes for levels, gradients and paged levels, and what it refuses (no GPU)."""
import struct
import sys

import pytest
import torch

import paper_2603_20586_b200.binding as mka


def _t(*shape, dtype=torch.bfloat16):
    return torch.zeros(*shape, dtype=dtype)


def _words(b):
    return struct.unpack(f"{len(b) // 8}q", b)


def test_levels_are_what_the_struct_holds():
    k = [_t(2, 3, 40, 64), None, _t(2, 3, 0, 64)]
    big = _t(2, 90, 3, 64)
    k[1], v = big.permute(0, 2, 1, 3), [_t(2, 3, 40, 64), torch.zeros_like(big).permute(0, 2, 1, 3), None]
    w = _words(mka._levels(k, v))
    assert w[:6] == (k[0].data_ptr(), v[0].data_ptr(), 40, *k[0].stride()[:3])
    assert w[6:12] == (k[1].data_ptr(), v[1].data_ptr(), 90, *k[1].stride()[:3]) and w[12:] == (0,) * 6
    assert _words(mka._levels((None, k[0], None), (None, v[0], None)))[:6] == (0,) * 6


@pytest.mark.parametrize("k,v", [
    (_t(2, 3, 40, 64), _t(2, 3, 41, 64)),                     # unlike shapes
    (_t(2, 3, 64, 40).transpose(2, 3), _t(2, 3, 64, 40).transpose(2, 3)),       # columns not dense
    (_t(2, 3, 40, 64), _t(2, 40, 3, 64).permute(0, 2, 1, 3)),  # unlike strides
    (_t(2, 3, 40, 64), None),
    (_t(3, 40, 64), _t(3, 40, 64)),
])
def test_levels_refuse(k, v):
    with pytest.raises(AssertionError):
        mka._levels([k, None, None], [v, None, None])


def test_paged_levels_are_what_the_struct_holds():
    pk, pv = _t(9, 2, 16, 64), _t(9, 2, 16, 64)
    tab, per_head, rows = _t(3, 4, dtype=torch.int32), _t(3, 2, 5, dtype=torch.int32), _t(3, dtype=torch.int32)
    w = _words(mka._paged_levels([pk, None, pk], [pv, None, pv], [tab, None, per_head], [rows, None, None], [60, 7, 33]))
    assert w[:12] == (pk.data_ptr(), pv.data_ptr(), tab.data_ptr(), rows.data_ptr(), 60, 4, 0, 16, *pk.stride()[:3], 9)
    assert w[12:24] == (0,) * 7 + (1, 0, 0, 0, 0)
    assert w[24:] == (pk.data_ptr(), pv.data_ptr(), per_head.data_ptr(), 0, 33, 10, 5, 16, *pk.stride()[:3], 9)
    assert _words(mka._paged_levels([pk] * 3, [pv] * 3, [tab] * 3, None, (1, 0, 2)))[12:24] == (0,) * 7 + (1, 0, 0, 0, 0)
    for bad_tab, bad_rows in ((tab.long(), rows), (tab, rows.long()), (tab[0], rows), (tab.t(), rows)):
        with pytest.raises(AssertionError):
            mka._paged_levels([pk, None, None], [pv, None, None], [bad_tab, None, None], [bad_rows, None, None], [60, 0, 0])


def test_outputs():
    q = _t(2, 3, 40, 64)
    assert mka._empty_f32(q, 3, 0).shape == (2, 3, 40) and mka._empty_f32(q, 2, 3).shape == (2, 3, 3)
    assert mka._empty_f32(q, 0, 0).shape == () and mka._empty_f32(q, 4, 0).dtype == torch.float32
    a, none = mka._host_args.empties_like([q, None])
    assert none is None and a.shape == q.shape and a.dtype == q.dtype and a.stride() == q.stride()


def test_what_answers_an_index_is_taken():
    k, v, tab = _t(2, 3, 40, 64), _t(2, 3, 40, 64), _t(3, 4, dtype=torch.int32)
    want = mka._levels([k, None, k], [v, None, v])
    assert mka._levels({0: k, 1: None, 2: k}, {0: v, 2: v}) == want and mka._levels([k, None, k, None], (v, None, v)) == want
    both = torch.stack([k, k, k])
    assert _words(mka._levels(both, both))[6] == both[1].data_ptr()
    with pytest.raises(IndexError):
        mka._levels([k], [v])


def test_rows_of_paged_levels_are_whole_numbers_by_value():
    pk, pv, tab = _t(9, 2, 16, 64), _t(9, 2, 16, 64), _t(3, 4, dtype=torch.int32)
    want = mka._paged_levels([pk, None, pk], [pv, None, pv], [tab, None, tab], None, [60, 0, 33])
    for n in ([60.0, None, 33.9], [torch.tensor(60), "absent", 33], {0: 60, 2: 33}):           # beside a pool of None nothing is looked at
        assert mka._paged_levels([pk, None, pk], [pv, None, pv], [tab, None, tab], None, n) == want
    with pytest.raises(TypeError):
        mka._paged_levels([pk, None, None], [pv, None, None], [tab, None, None], None, [None, 0, 0])


def test_gradients_follow_the_keys():
    k, g, h = _t(2, 3, 40, 64), _t(2, 3, 40, 64), _t(2, 3, 40, 64)
    w = _words(mka._host_args.grads([k, None, k[:, :, :0]], [g, g, None], [h, h, None]))
    assert w[:6] == (g.data_ptr(), h.data_ptr(), 40, *g.stride()[:3]) and w[6:] == (0,) * 12
    for dk, dv in ((None, h), (g, None), (g, h.transpose(2, 3)), (g.transpose(2, 3), h.transpose(2, 3))):
        with pytest.raises(AssertionError):                                                     # keys without room for their gradients
            mka._host_args.grads([k, None, None], [dk, None, None], [dv, None, None])


def test_module_of_another_torch_or_python_is_not_loaded(monkeypatch):
    from paper_2603_20586_b200 import build
    own = build.host_module()
    assert mka._host_args.__file__ == own and not build._stale(own, [build.HOST_SRC])
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".later")
    assert build.host_module() != own and build._stale(build.host_module(), [build.HOST_SRC])
    with pytest.raises(ImportError, match="later"):
        mka._load_host_args()
    monkeypatch.undo()
    monkeypatch.setattr(sys.implementation, "cache_tag", "cpython-999")
    assert build.host_module() != own
