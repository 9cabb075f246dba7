"""Keys that hold infinities, NaN or huge numbers in the score kernels: the log-sum-exp of a row is NaN where one of its logits is
NaN or +inf, and otherwise what the visible logits give, wherever in a tile such a key lies; the other keys keep their scores."""
import numpy as np
import pytest
import torch

from paper_2609_31395_b200 import binding as B
from paper_2609_31395_b200 import harness as H
from paper_2609_31395_b200 import synth

import parity_util as U

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
VALUES = [float("nan"), float("inf"), float("-inf"), 3e9]
POSITIONS = [0, 3, 300, 301, 511, 512, 700, 705, 1203, 1204, 1299]          # odd and even columns of every group of eight


def _instance(head_dim, group, window, causal, value, position, L=1300):
    wl = synth.Workload("special", 1, 2, group, [L], [window], [L // 3], head_dim=head_dim, causal=causal, seed=position + group)
    inst = synth.generate(wl, DEV)
    page = int(inst.page_table[0, position // wl.page_size])
    inst.pool[0, 0, page, position % wl.page_size, 0, 5] = value          # one element of one key of head 0
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads, H.sizes_of(inst),
                        want_lse=True)
    return wl, inst, comp


def _logits(wl, inst):
    """float64 [heads, rows, keys], -inf where a row does not see a key; a product with a special element as IEEE has it."""
    L, W, Hkv, G, P = wl.seq_lens[0], wl.windows[0], wl.n_kv_heads, wl.group, wl.page_size
    j = torch.arange(L, device=DEV)
    slots = inst.page_table[0].long()[j // P] * P + j % P
    k = inst.pool[0, 0].reshape(-1, Hkv, wl.head_dim)[slots].double().cpu().numpy().transpose(1, 0, 2)
    q = inst.q[0].view(W, Hkv, G, wl.head_dim).permute(1, 0, 2, 3).reshape(Hkv, W * G, wl.head_dim).double().cpu().numpy()
    with np.errstate(invalid="ignore"):
        s = q @ k.transpose(0, 2, 1) * wl.sm_scale
    if wl.causal:
        last = L - W + np.repeat(np.arange(W), G)
        s[:, np.arange(L)[None, :] > last[:, None]] = -np.inf
    return s


LAYOUTS = [(128, 4, 5, True, 0), (96, 3, 30, False, 0), (128, 4, 40, True, 1), (64, 8, 64, False, 1), (128, 8, 20, False, 1)]
# (the tcgen05 kernel, path 1, keeps its reference to 24 bits: logits beyond 2^31 are out of its range)
LSE_CASES = [layout + (value,) for layout in LAYOUTS for value in VALUES + ([1e30] if layout[4] == 0 else [])]


@pytest.mark.parametrize("head_dim,group,window,causal,path,value", LSE_CASES)
def test_lse(head_dim, group, window, causal, path, value):
    for position in POSITIONS:
        wl, inst, comp = _instance(head_dim, group, window, causal, value, position)
        assert B.actkv_score_path(comp.pd, wl.n_q_heads, window, wl.sm_scale, inst.q) == path
        s = _logits(wl, inst)
        comp.run_score(inst.q, inst.win_indptr, inst.tok_indptr, wl.sm_scale, causal)
        torch.cuda.synchronize()
        comp.check_status()
        got = comp.lse.cpu().numpy()[0].reshape(window, wl.n_kv_heads, group).transpose(1, 0, 2).reshape(wl.n_kv_heads, -1)
        with np.errstate(invalid="ignore"):
            top = s.max(axis=2, keepdims=True)
            want = np.log(np.exp(s - top).sum(axis=2)) + top[..., 0]
        assert np.array_equal(np.isnan(got), np.isnan(want)), position
        m = ~np.isnan(want)
        # a fp32 dot product (2^-20 of a huge one) and, where an exponential is a polynomial, 7.5e-5 of it
        assert (np.abs(got[m] - want[m]) <= 1e-4 + 2e-6 * np.abs(want[m])).all(), position


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("head_dim,group,window,causal,path", [(128, 4, 5, True, 0), (96, 3, 30, False, 0), (64, 1, 3, False, 0)])
def test_pooled_score(head_dim, group, window, causal, path, value):
    """The other keys' scores do not depend on such a key; its own: +inf logits count as inf, NaN and -inf ones as nothing."""
    for position in POSITIONS:
        wl, inst, comp = _instance(head_dim, group, window, causal, value, position)
        assert B.actkv_score_path(comp.pd, wl.n_q_heads, window, wl.sm_scale, inst.q) == path
        s = _logits(wl, inst)
        lse = np.full((1, window, wl.n_q_heads), 8.0, dtype=np.float32)
        comp.run_score(inst.q, inst.win_indptr, inst.tok_indptr, wl.sm_scale, causal, lse_in=torch.from_numpy(lse).to(DEV))
        torch.cuda.synchronize()
        comp.check_status()
        with np.errstate(over="ignore"):
            a = np.nan_to_num(np.exp(np.where(s > -np.inf, s, -np.inf) - 8.0), nan=0.0, posinf=np.inf)
        want = a.reshape(wl.n_kv_heads, window, group, -1).max(axis=2).sum(axis=1) / window
        got = comp.score.cpu().numpy()[0]
        big = want > 3e38
        assert np.array_equal(np.isinf(got), big) and not np.isnan(got).any(), position
        assert (np.abs(got[~big] - want[~big]) <= U.SCORE_RTOL * want[~big] + 1e-30).all(), position
