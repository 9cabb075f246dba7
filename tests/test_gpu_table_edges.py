"""Compaction plans and table updates at the edges of how they are split over CTAs (256 requests per scan, 1024 table
entries per CTA) and pages copied in parts, against the oracle on every byte of pool, tables and free list."""
import numpy as np
import pytest
import torch

from oracle import actkv_oracle as O
from paper_2609_31395_b200 import binding as B

import parity_util as U
import test_gpu_compact_inplace as TI
from test_gpu_random_compact import _check_fresh, _fresh_page_oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _lens(kind, rng):
    if kind == "many requests":                    # more than a CTA scans in one round; some stay as they are
        lens = [int(x) for x in rng.integers(1, 41, 300)]
        return lens, [int(rng.choice([0, 1, max(1, L // 3), L, L + 2])) for L in lens]
    if kind == "long tables":                      # 1023 .. 2250 pages of 4 tokens
        lens = [4092, 4096, 4097, 9000]
        return lens, [4000, 1, 4096, 5000]
    return [700, 90], [130, 33]                    # few pages: each is copied in parts


@pytest.mark.parametrize("form", ["fresh pages", "fresh pages, no status word", "no workspace", "in place"])
@pytest.mark.parametrize("kind", ["many requests", "long tables", "page parts"])
def test_edges(kind, form):
    rng = np.random.default_rng(11)
    lens, budgets = _lens(kind, rng)
    P, Hkv, D, NL = (32, 3, 72, 1) if kind == "page parts" else (4, 1, 64, 2)
    inst, sel, ki, stride, max_keep = TI._direct_case(rng, lens, budgets, P, Hkv, D, NL)
    pool_before, tables_before = U.bits(inst.pool), U.oracle_tables(inst)
    pd = B.pool_desc(inst.pool)
    td = B.tables_desc(inst.page_table, inst.seq_len, inst.free_list, inst.free_count)
    d_sel, d_ki = torch.from_numpy(sel).to(DEV), torch.from_numpy(ki).to(DEV)
    d_bud = torch.tensor(budgets, dtype=torch.int32, device=DEV)
    status = None if "no status" in form else torch.zeros(4, dtype=torch.int32, device=DEV)
    if form == "in place":
        d_order = torch.full_like(d_sel, -9)
        B.actkv_compact_inplace(pd, td, 0, NL, d_sel, stride, d_ki, d_bud, max_keep, d_order, status)
        torch.cuda.synchronize()
        assert status.cpu().tolist()[0] == 0
        TI._check_against_oracle(inst, pool_before, tables_before, sel, ki, budgets, d_order.cpu().numpy())
        return
    want_pool, want_t = _fresh_page_oracle(inst, pool_before, tables_before, sel, ki, budgets, NL)
    if form == "no workspace":
        B.actkv_compact_noalloc(pd, td, 0, NL, d_sel, stride, d_ki, d_bud, max_keep, status)
    else:
        ws = torch.empty(B.actkv_compact_workspace_bytes(len(lens), td.max_pages), dtype=torch.uint8, device=DEV)
        B.actkv_compact(pd, td, 0, NL, d_sel, stride, d_ki, d_bud, max_keep, ws, status)
    torch.cuda.synchronize()
    assert status is None or status.cpu().tolist()[0] == 0
    _check_fresh(inst, want_pool, want_t)


@pytest.mark.parametrize("which", ["old page", "free page"])
def test_a_page_id_out_of_range_met_by_any_cta_of_the_plan(which):
    """The bad id lies in the last request's last table entries, far from what the first CTA reads."""
    rng = np.random.default_rng(12)
    lens, budgets = [900, 4500, 8200], [300, 4200, 4500]
    inst, sel, ki, stride, max_keep = TI._direct_case(rng, lens, budgets, 4, 1, 64, 1)
    fc = int(inst.free_count.cpu())
    if which == "old page":
        inst.page_table[2, 2040] = inst.pool.shape[2] + 7
    else:
        inst.free_list[fc - 1 - (75 + 1050 + 1100)] = -3       # the 1100th page that request 2 pops
    snap = [U.bits(inst.pool).copy()] + [t.clone() for t in (inst.page_table, inst.seq_len, inst.free_list, inst.free_count)]
    pd = B.pool_desc(inst.pool)
    td = B.tables_desc(inst.page_table, inst.seq_len, inst.free_list, inst.free_count)
    d_sel, d_ki = torch.from_numpy(sel).to(DEV), torch.from_numpy(ki).to(DEV)
    d_bud = torch.tensor(budgets, dtype=torch.int32, device=DEV)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.actkv_compact_deferred_workspace_bytes(pd, 3, td.max_pages, 1, max_keep), dtype=torch.uint8, device=DEV)
    for call in ("one", "two"):
        status.zero_()
        if call == "one":
            B.actkv_compact(pd, td, 0, 1, d_sel, stride, d_ki, d_bud, max_keep, ws, status)
        else:
            B.actkv_compact_begin(pd, td, 0, 1, d_sel, stride, d_ki, d_bud, max_keep, ws, status)
            B.actkv_compact_end(pd, td, 0, 1, d_sel, stride, d_ki, d_bud, max_keep, ws, status)
        torch.cuda.synchronize()
        assert status.cpu().tolist()[0] == B.E_BADPAGE
        assert np.array_equal(U.bits(inst.pool), snap[0])
        for t, s in zip((inst.page_table, inst.seq_len, inst.free_list, inst.free_count), snap[1:]):
            assert torch.equal(t, s)


@pytest.mark.parametrize("counts", [[1], [1023, 1], [1024, 1025, 0, 7], [0, 0, 5000], [3] * 700])
def test_gather_over_request_boundaries(counts):
    """1024 survivors per CTA; requests that keep nothing; many requests inside one CTA."""
    rng = np.random.default_rng(len(counts))
    lens = [c + int(rng.integers(1, 9)) for c in counts]
    tok = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    ki = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    n_outer, total = 3, int(ki[-1])
    sel = np.full((n_outer, total + 2), -1, dtype=np.int32)
    src = rng.random((n_outer, int(tok[-1])), dtype=np.float32)
    want = np.zeros((n_outer, total + 1), dtype=np.float32)
    for o in range(n_outer):
        for r, c in enumerate(counts):
            pick = rng.permutation(lens[r])[:c]
            sel[o, ki[r]:ki[r + 1]] = pick
            want[o, ki[r]:ki[r + 1]] = src[o, tok[r] + pick]
    dst = torch.zeros((n_outer, total + 1), device=DEV)
    B.actkv_gather_f32(torch.from_numpy(src).to(DEV), src.shape[1], torch.from_numpy(tok).to(DEV), torch.from_numpy(sel).to(DEV),
                       sel.shape[1], torch.from_numpy(ki).to(DEV), n_outer, len(counts), total + 1, dst, total + 1)
    torch.cuda.synchronize()
    assert np.array_equal(dst.cpu().numpy(), want)


def test_gather_takes_all_survivors_whatever_the_bound():
    n, L = 5000, 6000
    sel = np.sort(np.random.default_rng(3).permutation(L)[:n]).astype(np.int32)
    src = np.random.default_rng(4).random((1, L), dtype=np.float32)
    dst = torch.zeros((1, n), device=DEV)
    i32 = lambda *v: torch.tensor(v, dtype=torch.int32, device=DEV)  # noqa: E731
    B.actkv_gather_f32(torch.from_numpy(src).to(DEV), L, i32(0, L), torch.from_numpy(sel[None]).to(DEV), n, i32(0, n), 1, 1, 100, dst, n)
    torch.cuda.synchronize()
    assert np.array_equal(dst.cpu().numpy()[0], src[0, sel])


@pytest.mark.parametrize("lens,budgets", [([256, 257, 511, 513, 2], [128, 256, 257, 512, 1]), ([40000], [39990]),
                                          ([9000, 3000], [4500, 2999])])
def test_inplace_slots_over_cta_boundaries(lens, budgets):
    """Regions of one slot more or less than the 128 and 256 slots of a CTA, one whose list takes several rounds of the
    32-way search, one whose region is nearly everything; enough heads for either launch shape."""
    for Hkv, NL in ((1, 1), (8, 3)):
        rng = np.random.default_rng(5)
        inst, sel, ki, stride, max_keep = TI._direct_case(rng, lens, budgets, 16, Hkv, 64, NL)
        pool_before, tables_before = U.bits(inst.pool), U.oracle_tables(inst)
        d_sel = torch.from_numpy(sel).to(DEV)
        d_order = torch.full_like(d_sel, -9)
        status = torch.zeros(4, dtype=torch.int32, device=DEV)
        B.actkv_compact_inplace(B.pool_desc(inst.pool), B.tables_desc(inst.page_table, inst.seq_len, inst.free_list, inst.free_count),
                                0, NL, d_sel, stride, torch.from_numpy(ki).to(DEV),
                                torch.tensor(budgets, dtype=torch.int32, device=DEV), max_keep, d_order, status)
        torch.cuda.synchronize()
        assert status.cpu().tolist()[0] == 0
        TI._check_against_oracle(inst, pool_before, tables_before, sel, ki, budgets, d_order.cpu().numpy())
