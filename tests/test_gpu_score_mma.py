"""The warp-level (mma.sync) score kernels against the oracle at the edges of their tiling: key tiles of 16 or 32, four
warps per CTA, chunks of 64 rows, CTA ranges of up to 2048 keys, head dimensions that are no multiple of 32, groups
padded to a power of two, pages whose size is not a power of two, a negative softmax scale."""
import numpy as np
import pytest
import torch

from oracle import actkv_oracle as O
from paper_2609_31395_b200 import binding as B
from paper_2609_31395_b200 import harness as H
from paper_2609_31395_b200 import synth

import parity_util as U

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

#        head_dim, page, group, window, lengths
CASES = [(128, 16, 1, 1, [1, 15, 16, 17, 31, 33]),
         (128, 16, 4, 15, [127, 128, 129, 2047, 2049, 4500]),
         (64, 16, 2, 31, [64, 511, 513]),
         (8, 16, 3, 5, [40, 700]),
         (96, 16, 16, 5, [300, 2100]),
         (136, 16, 32, 3, [17, 1000]),
         (256, 16, 7, 9, [255, 257]),
         (128, 12, 8, 8, [95, 97, 2051]),
         (200, 24, 5, 13, [47, 900])]


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("head_dim,page,group,window,lens", CASES)
def test_edges(head_dim, page, group, window, lens, causal):
    wins = [min(window, L) for L in lens]
    wl = synth.Workload("mma", 2, 2, group, lens, wins, [max(1, L // 3) for L in lens], head_dim=head_dim, page_size=page,
                        causal=causal, table_style="fragmented", seed=head_dim + group, poison_tail=True)
    inst = synth.generate(wl, DEV)
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads,
                        H.sizes_of(inst), want_lse=True)
    for scale in (wl.sm_scale, -wl.sm_scale):
        assert B.actkv_score_path(comp.pd, wl.n_q_heads, max(wins), scale, inst.q) == 0
        want, lse, _ = O.score(U.bits(inst.pool), inst.page_table.cpu().numpy(), inst.seq_len.cpu().numpy(), U.bits(inst.q),
                               inst.win_indptr.cpu().numpy(), wl.n_q_heads, scale, causal)
        comp.score.fill_(float("nan"))
        comp.run_score(inst.q, inst.win_indptr, inst.tok_indptr, scale, causal)
        torch.cuda.synchronize()
        comp.check_status()
        got = comp.score.cpu().numpy()
        assert np.isfinite(got).all()
        assert U.max_rel(got, want) <= U.SCORE_RTOL
        # fp32 dot products of up to 256 bf16 numbers: 256 2^-24 of sums of order 10
        assert np.abs(comp.lse.cpu().numpy() - lse)[~np.isnan(lse)].max() < 1e-4
