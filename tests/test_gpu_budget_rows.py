"""Token confidence at the edges of its two forms (a cluster of 1, 2, 4 or 8 CTAs per row, one CTA per row) and of the
trend's phases, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2609_31395_b200 import binding as B

from test_gpu_budget import DEV, _compare

pytestmark = pytest.mark.gpu


def _logits(rows, vocab, kind, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    z = 3.0 * torch.randn((rows, vocab), generator=g, device=DEV)
    if kind == "equal":
        z.fill_(-1.25)                                     # every logit a candidate: the lists overflow
    elif kind == "masked":
        z[torch.rand(z.shape, generator=g, device=DEV) < 0.97] = float("-inf")
    elif kind == "ascending":
        z = z.sort(dim=1).values.contiguous()
    elif kind == "peak":
        z[:, vocab // 2] = 60.0
    return z


def _run(rows, vocab, kind, k, reqs):
    cut = sorted({0, rows} | {rows * i // reqs for i in range(reqs + 1)})
    reqs = len(cut) - 1
    tok = torch.tensor(cut, dtype=torch.int32, device=DEV)
    params = B.BudgetParams.paper_defaults()
    params.k = k
    hist = torch.zeros((reqs, 100 + rows), dtype=torch.float32)
    _compare(_logits(rows, vocab, kind, vocab + rows), tok, hist, torch.zeros(reqs, dtype=torch.int32),
             torch.full((reqs,), 512, dtype=torch.int32), params)


@pytest.mark.parametrize("vocab", [2, 31, 1000, 8183, 8186, 8187, 16381, 32003, 65537, 131073])
def test_rows_of_a_few(vocab):
    _run(3, vocab, "normal", min(20, vocab), 2)           # odd lengths: the rows start at every alignment


@pytest.mark.parametrize("kind", ["equal", "masked", "ascending", "peak"])
@pytest.mark.parametrize("rows", [2, 75])                 # 75 rows x 8 CTAs is past the cluster form's limit
def test_distributions(kind, rows):
    _run(rows, 40001, kind, 20, 5)


@pytest.mark.parametrize("k", [1, 63, 64, 65, 300])
def test_k(k):
    _run(2, 20000, "normal", k, 1)


@pytest.mark.parametrize("w,s,length", [(64, 8, 64), (64, 8, 71), (64, 8, 72), (64, 8, 2600), (64, 1, 5000), (10, 3, 900), (1, 1, 300),
                                         (64, 8, 40000)])
def test_trend(w, s, length):
    g = torch.Generator().manual_seed(length + w)
    hist = 4.0 + torch.rand((2, length), generator=g)
    params = B.BudgetParams.paper_defaults()
    params.w, params.s = w, s
    tok = torch.zeros(3, dtype=torch.int32, device=DEV)
    _compare(torch.zeros((0, 16), device=DEV), tok, hist, torch.tensor([length, max(0, length - 5)], dtype=torch.int32),
             torch.tensor([512, 700], dtype=torch.int32), params)


@pytest.mark.parametrize("n", [3, 5, 64, 255, 256, 257, 999, 4000])
def test_a_slope_of_zero_is_zero(n):
    """Histories that read the same backwards: the slope is 0 and the budgets stay.  One with an infinite confidence has none."""
    R = 9
    params = B.BudgetParams.paper_defaults()
    params.w = params.s = 1
    params.b_percent = 100.0
    g = torch.Generator().manual_seed(n)
    hist = 1.0 + 8.0 * torch.rand((R, n), generator=g)
    hist[0] = 4.0
    hist[0, n // 2] = 4.25                                 # (an even n: not symmetric, falls or rises)
    hist[1] = (hist[1] * 4).round() / 4
    hist[1:] = torch.where(torch.arange(n) < (n + 1) // 2, hist[1:], hist[1:].flip(1))
    hist[8, 0] = float("inf")
    i32 = lambda v: torch.full((R,), v, dtype=torch.int32, device=DEV)  # noqa: E731
    out, slope, status = i32(0), torch.full((R,), 7.0, dtype=torch.float64, device=DEV), torch.zeros(4, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.actkv_budget_workspace_bytes(0, R, n), dtype=torch.uint8, device=DEV)
    B.actkv_budget(None, None, 0, 16, hist.to(DEV), i32(n), n, params, None, i32(512), out, slope, R, ws, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    slope, out = slope.cpu(), out.cpu()
    zero = slice(0, 8) if n % 2 else slice(1, 8)
    assert (slope[zero] == 0).all() and (out[zero] == 512).all()
    assert torch.isnan(slope[8]) and out[8] == 512
