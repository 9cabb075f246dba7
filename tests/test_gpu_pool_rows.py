"""The pooled-score kernel where its layouts change: rows around 16 (narrow fold), 64 (LSE in the contraction), 128, 256 and
512, at both head dimensions, alone and as windows of different length in one launch; rows whose supplied LSE is infinite."""
import numpy as np
import pytest
import torch

from oracle import actkv_oracle as O
from paper_2609_31395_b200 import harness as H
from paper_2609_31395_b200 import synth

import parity_util as U

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(wl, spoil=False):
    inst = synth.generate(wl, DEV)
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads, H.sizes_of(inst))
    args = (U.bits(inst.pool), inst.page_table.cpu().numpy(), inst.seq_len.cpu().numpy(), U.bits(inst.q),
            inst.win_indptr.cpu().numpy(), wl.n_q_heads, wl.sm_scale, wl.causal)
    _, lse, _ = O.score(*args)
    lse = np.nan_to_num(lse).astype(np.float32)
    if spoil:
        lse[:, ::3, ::2] = np.inf                       # such a row takes part in no maximum
    want, _, _ = O.score(*args, lse_in=lse)
    comp.score.fill_(float("nan"))
    comp.run_score(inst.q, inst.win_indptr, inst.tok_indptr, wl.sm_scale, wl.causal, lse_in=torch.from_numpy(lse).to(DEV))
    torch.cuda.synchronize()
    comp.check_status()
    got = comp.score.cpu().numpy()
    assert np.isfinite(got).all()
    m = want > 1e-30
    assert U.max_rel(got[m], want[m]) <= U.SCORE_RTOL and np.abs(got[~m]).max(initial=0.0) <= 1e-30


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("group,windows", [(4, [16, 17]), (4, [32, 33, 16]), (4, [64, 65]), (8, [64, 8, 33]), (8, [33, 32, 31]),
                                           (2, [200, 33, 64, 129]), (1, [65, 64, 300]), (7, [20, 9]), (32, [3, 8, 9]), (16, [5, 33])])
def test_rows(group, windows, head_dim, causal):
    lens = [700 + 131 * i for i in range(len(windows))]
    _check(synth.Workload("rows", 2, 2, group, lens, windows, [L // 3 for L in lens], head_dim=head_dim, causal=causal,
                          table_style="fragmented", seed=group + head_dim, poison_tail=True))


@pytest.mark.parametrize("head_dim,windows", [(64, [64, 10]), (128, [32, 20]), (128, [64, 64])])
def test_rows_with_an_infinite_lse(head_dim, windows):
    _check(synth.Workload("inf", 1, 2, 8, [500, 300], windows, [100, 50], head_dim=head_dim, table_style="fragmented", seed=3),
           spoil=True)


@pytest.mark.parametrize("head_dim,group,windows", [(64, 8, [64, 20]), (64, 4, [128, 90]), (128, 4, [64, 40]), (128, 8, [32, 9]),
                                                    (128, 1, [200, 70]), (64, 16, [32, 5])])
def test_scores_are_not_rounded_to_one_side(head_dim, group, windows):
    """The mean relative error against float64.  Sums rounded to nearest have next to none; sums of magnitude 8 to 16 (in log2
    units) rounded towards zero make a score up to 2^-20 ln 2 = 6.6e-7 too large, half of that on average."""
    lens = [3000, 1700]
    wl = synth.Workload("bias", 2, 4, group, lens, windows, [L // 3 for L in lens], head_dim=head_dim, table_style="fragmented",
                        seed=head_dim)
    inst = synth.generate(wl, DEV)
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads, H.sizes_of(inst))
    args = (U.bits(inst.pool), inst.page_table.cpu().numpy(), inst.seq_len.cpu().numpy(), U.bits(inst.q),
            inst.win_indptr.cpu().numpy(), wl.n_q_heads, wl.sm_scale, False)
    lse = O.score(*args)[1].astype(np.float32)
    want = O.score(*args, lse_in=lse)[0]
    comp.run_score(inst.q, inst.win_indptr, inst.tok_indptr, wl.sm_scale, False, lse_in=torch.from_numpy(lse).to(DEV))
    torch.cuda.synchronize()
    comp.check_status()
    rel = comp.score.cpu().numpy().astype(np.float64) / want - 1.0
    assert abs(rel.mean()) < 1e-7 and np.abs(rel).max() < 3e-6


def test_a_softmax_scale_whose_inverse_overflows():
    """Every logit is next to 0 then, and a score is what the supplied LSEs say."""
    wl = synth.Workload("scale", 1, 2, 4, [300, 200], [40, 30], [100, 50], table_style="fragmented", seed=1)
    inst = synth.generate(wl, DEV)
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads, H.sizes_of(inst))
    lse = np.random.default_rng(0).uniform(-20.0, 20.0, (1, 70, 8)).astype(np.float32)
    comp.run_score(inst.q, inst.win_indptr, inst.tok_indptr, 2e-38, False, lse_in=torch.from_numpy(lse).to(DEV))
    torch.cuda.synchronize()
    comp.check_status()
    got = comp.score.cpu().numpy()[0]
    a = np.exp(-lse[0].astype(np.float64)).reshape(70, 2, 4).max(axis=2)
    for r, (w0, w1, t0, t1) in enumerate([(0, 40, 0, 300), (40, 70, 300, 500)]):
        want = a[w0:w1].mean(axis=0)
        assert (np.abs(got[:, t0:t1] / want[:, None] - 1.0) < U.SCORE_RTOL).all(), r
