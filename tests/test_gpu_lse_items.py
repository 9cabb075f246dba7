"""LSE pass at the edges of its work items: rows around half a block and a block, groups that do not divide 64, several row groups,
chunks of the shortest length, requests that end early; against float64, and the same bits on every run."""
import random

import pytest
import torch

from paper_2609_31395_b200 import binding as B
from paper_2609_31395_b200 import harness as H
from paper_2609_31395_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _lse64(b, window_left=0):
    wl = b.wl
    G, D, P, Hkv = wl.group, wl.head_dim, wl.page_size, wl.n_kv_heads
    out, w0 = [], 0
    for r, (L, W) in enumerate(zip(wl.seq_lens, wl.windows)):
        j = torch.arange(L, device=DEV)
        slots = b.page_table[r].long()[j // P] * P + j % P
        k = b.pool[:, 0].reshape(wl.n_layers, -1, Hkv, D)[:, slots].permute(0, 2, 3, 1).double()          # [NL, Hkv, D, L]
        q = b.q[:, w0:w0 + W].view(wl.n_layers, W, Hkv, G, D).permute(0, 2, 1, 3, 4).reshape(wl.n_layers, Hkv, W * G, D).double()
        s = (q @ k) * wl.sm_scale
        last = (L - W if wl.causal else L - 1) + torch.arange(W, device=DEV).repeat_interleave(G) * int(wl.causal)
        s.masked_fill_(j[None, :] > last[:, None], float("-inf"))
        if window_left:
            s.masked_fill_(j[None, :] <= last[:, None] - window_left, float("-inf"))
        out.append(s.logsumexp(-1).view(wl.n_layers, Hkv, W, G).permute(0, 2, 1, 3).reshape(wl.n_layers, W, Hkv * G))
        w0 += W
    return torch.cat(out, 1)


@pytest.mark.parametrize("group,windows,head_dim,causal", [
    (4, [16, 17, 32, 33, 48, 49, 64], 128, True),        # 64, 68, 128, 132, 192, 196, 256 rows
    (4, [80, 81, 112, 113, 128], 128, False),            # 320, 324, 448, 452, 512: both halves of the Q columns
    (8, [8, 9, 24, 25, 56, 64], 64, True),               # four blocks in one half
    (7, [9, 10, 18, 19, 40, 73], 128, True),             # groups across the edges of half blocks; 511 rows are two row groups
    (32, [2, 3, 5, 20], 64, False),
    (5, [13, 26, 27, 110], 128, True),                   # 550 rows
])
def test_rows_around_the_edges_of_items(group, windows, head_dim, causal):
    lens = [max(w, n) for w, n in zip(windows, [700, 129, 2600, 512, 1, 1537, 300])]
    wl = synth.Workload("items", 2, 2, group, lens, windows, [max(1, n // 4) for n in lens], head_dim=head_dim, causal=causal,
                        table_style="fragmented", seed=61)
    b = synth.generate(wl, DEV)
    comp = H.Compressor(b.pool, b.page_table, b.seq_len, b.free_list, b.free_count, wl.n_q_heads, H.sizes_of(b), want_lse=True)
    runs = []
    for _ in range(4):
        comp.lse.fill_(float("nan"))
        comp.run_lse(b.q, b.win_indptr, b.tok_indptr, wl.sm_scale, wl.causal, 0, wl.n_layers, comp.lse)
        runs.append(comp.lse.clone())
    comp.check_status()
    # one exponential in eight is a cubic of relative error 7.5e-5; float32 dot products of 128 terms add 1e-5
    assert (runs[0].double() - _lse64(b)).abs().max() < 1e-4
    for x in runs[1:]:
        assert torch.equal(x, runs[0])


@pytest.mark.parametrize("head_dim", [128, 64])
@pytest.mark.parametrize("max_rows", [384, 800])
def test_items_of_one_to_three_blocks_in_turn(max_rows, head_dim):
    # an item of three blocks takes Q columns of both halves at head_dim 128: every order of items of different widths in one CTA
    rows = [n for n in (260, 384, 64, 320, 256, 324, 128, 192, 388, 512, 516, 640, 644, 768, 772, 800) if n <= max_rows]
    windows = [n // 4 for n in rows + rows[::-1]]
    lens = [max(w, 130 + 67 * i) for i, w in enumerate(windows)]
    wl = synth.Workload("blocks", 8, 4, 4, lens, windows, [n // 4 for n in lens], head_dim=head_dim, causal=True,
                        table_style="fragmented", seed=73)
    b = synth.generate(wl, DEV)
    comp = H.Compressor(b.pool, b.page_table, b.seq_len, b.free_list, b.free_count, wl.n_q_heads, H.sizes_of(b), want_lse=True)
    runs = []
    for _ in range(3):
        comp.lse.fill_(float("nan"))
        comp.run_lse(b.q, b.win_indptr, b.tok_indptr, wl.sm_scale, wl.causal, 0, wl.n_layers, comp.lse)
        runs.append(comp.lse.clone())
    comp.check_status()
    assert (runs[0].double() - _lse64(b)).abs().max() < 1e-4        # (the cubic and float32 dot products, as above)
    assert torch.equal(runs[1], runs[0]) and torch.equal(runs[2], runs[0])


@pytest.mark.parametrize("group,windows,lens,head_dim,causal", [
    (4, [32], [4096], 128, False),                       # one item of rows, eight chunks
    (4, [64, 17], [1500, 129], 128, True),               # a full item, and one of 68 rows
    (8, [64], [300], 64, True),                          # 512 rows, one chunk: two items side by side
    (7, [19, 9], [700, 513], 128, True),                 # 133 and 63 rows
    (16, [40], [2000], 64, False),                       # 640 rows: two launches of the pooled-score pass
])
def test_launches_that_leave_sms_idle(group, windows, lens, head_dim, causal):
    wl = synth.Workload("few", 1, 2, group, lens, windows, [max(1, n // 4) for n in lens], head_dim=head_dim, causal=causal,
                        table_style="fragmented", seed=67)
    b = synth.generate(wl, DEV)
    args = (b.q, b.win_indptr, b.tok_indptr, wl.sm_scale, wl.causal, 0, 1)
    comp = H.Compressor(b.pool, b.page_table, b.seq_len, b.free_list, b.free_count, wl.n_q_heads, H.sizes_of(b), want_lse=True)
    lse = torch.full_like(comp.lse, float("nan"))
    comp.run_lse(*args, lse)
    assert (lse.double() - _lse64(b)).abs().max() < 1e-4        # (the cubic and float32 dot products, as above)
    comp.run_score(*args, lse_in=lse)
    want = comp.score.clone()
    # both passes in one call: the same bits as one after the other
    comp.lse.fill_(float("nan"))
    comp.score.fill_(float("nan"))
    comp.run_score(*args)
    comp.check_status()
    assert torch.equal(comp.lse, lse) and torch.equal(comp.score, want)
    comp.lse = None                                             # nobody asks for the LSE: it goes to the workspace
    comp.score.fill_(float("nan"))
    comp.run_score(*args)
    assert torch.equal(comp.score, want)


@pytest.mark.parametrize("group,head_dim,causal,window_left", [
    (7, 128, True, 0), (7, 64, False, 0), (5, 128, False, 0), (3, 64, True, 150), (24, 128, True, 0), (4, 128, True, 0), (8, 64, False, 200),
])
def test_lanes_without_a_row_change_nothing(group, head_dim, causal, window_left):
    """More than three items per SM, so that every CTA goes on to others; keys of norm 40, of which one in place of a query makes logits
    beyond 2^40, and NaN behind the end of every request."""
    rng = random.Random(group)
    n_req = 20
    lens = [rng.randrange(130, 1000) for _ in range(n_req)]
    windows = [max(1, min(n, rng.randrange(66, 400) // group)) for n in lens]
    windows[0] = -(-66 // group)
    wl = synth.Workload("lanes", 6, 4, group, lens, windows, [max(1, n // 4) for n in lens], head_dim=head_dim, causal=causal,
                        table_style="fragmented", seed=71, poison_tail=True)
    b = synth.generate(wl, DEV)
    b.pool[:, 0] *= 40 / head_dim ** 0.5
    comp = H.Compressor(b.pool, b.page_table, b.seq_len, b.free_list, b.free_count, wl.n_q_heads, H.sizes_of(b), want_lse=True)
    z = comp.sz

    def lse():
        comp.lse.fill_(float("nan"))
        B.actkv_score_sliding(comp.pd, comp.td, 0, wl.n_layers, b.q, b.win_indptr, wl.n_q_heads, None, wl.sm_scale, wl.causal,
                              window_left, b.tok_indptr, comp.score, comp.lse, z.sum_win, z.max_win, z.sum_tok, z.max_tok,
                              comp.ws_score, comp.status)
        comp.check_status()
        return comp.lse.clone()

    first = lse()
    want = _lse64(b, window_left)
    # (the cubic as above; logits of up to 60 as float32 sums of 128 products)
    assert (first.double() - want).abs().max() < 1e-4 + 60 * 2.0 ** -20
    for _ in range(3):
        assert torch.equal(lse(), first)
    for r, n in enumerate(lens):                                # other bytes in the slots behind the end
        if n % wl.page_size:
            tail = b.pool[:, :, int(b.page_table[r, n // wl.page_size]), n % wl.page_size:]
            tail.copy_(torch.randn_like(tail.float()) * 100)
    assert torch.equal(lse(), first)
    rows = torch.repeat_interleave(torch.arange(n_req, device=DEV), torch.tensor(windows, device=DEV))
    b.q[:, rows % 2 == 1] = float("nan")                        # other queries beside every second request's
    assert torch.equal(lse()[:, rows % 2 == 0], first[:, rows % 2 == 0])
