"""Recall with the bank spread over a cluster: lists against the oracle, bit for bit, with many ties at the cut (few code bits), banks
that leave some CTAs without chunks, and lists longer than the bank."""
import numpy as np
import pytest
import torch

from mka_inputs import RecallConfig, make_recall

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


CASES = [
    RecallConfig("c_ties", 91, 2, 4, 2, 64, 9001, 2, 32, 64, len_frac=(1.0, 0.21)),
    RecallConfig("c_64", 92, 3, 8, 2, 64, 4097, 2, 64, 8, len_frac=(1.0, 0.004, 0.0)),
    RecallConfig("c_128", 93, 1, 2, 2, 128, 7000, 1, 128, 16),
    RecallConfig("c_256", 94, 1, 4, 4, 64, 1500, 2, 256, 5),
    RecallConfig("c_many", 95, 40, 2, 2, 64, 1100, 1, 64, 4, len_frac=(1.0, 0.5)),          # too many lists for clusters
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_recall_lists_are_bit_exact(mka, orc, cfg):
    P = make_recall(cfg, "cuda")
    codes = mka.mka_l3_index(P["pool_k"], P["proj"])
    table, n_sel, rows = mka.mka_l3_retrieve(P["q"], cfg.H_kv, P["proj"], codes, P["bank"], P["bank_len"], cfg.R, cfg.page_rows)
    t_ref, n_ref = orc.l3_retrieve(P["q"].float().cpu().numpy(), P["proj"].cpu().numpy(), codes.cpu().numpy().view(np.uint32),
                                   P["bank"].cpu().numpy(), P["bank_len"].cpu().numpy(), cfg.R, cfg.H_kv)
    assert np.array_equal(table.cpu().numpy(), t_ref)
    assert np.array_equal(n_sel.cpu().numpy(), n_ref) and np.array_equal(rows.cpu().numpy(), n_ref * cfg.page_rows)
