"""TopK and the fused keep-score + TopK where their histograms, rankings and CTA shapes can go wrong: lengths around the
limits of the CTA shapes and of the shared-memory copy, score sets that need one or many histogram levels, ties by the
hundred at the threshold, protected prefixes around the budget."""
import numpy as np
import pytest
import torch

from oracle import actkv_oracle as O
from paper_2609_31395_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _scores(kind, shape, rng):
    if kind == "equal":
        return np.full(shape, 0.25, dtype=np.float32)
    if kind == "zeros and ones":
        return (rng.random(shape) < 0.3).astype(np.float32)
    if kind == "few values":
        return (rng.integers(0, 7, shape) / 7.0).astype(np.float32)
    if kind == "one outlier":                              # the range is wide, nearly all keys share the lowest bin
        x = (1e-6 + 1e-9 * rng.random(shape)).astype(np.float32)
        x[..., shape[-1] // 2] = 200.0
        return x
    if kind == "subnormal":
        return (rng.random(shape) * 1e-40).astype(np.float32)
    return np.exp(2.0 * rng.standard_normal(shape)).astype(np.float32) / 4096.0


def _case(kind, lens, budgets, n_outer, seed):
    rng = np.random.default_rng(seed)
    tok = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    keep = [min(b, L) for b, L in zip(budgets, lens)]
    ki = np.concatenate([[0], np.cumsum(keep)]).astype(np.int32)
    sc = np.concatenate([_scores(kind, (n_outer, L), rng) for L in lens], axis=1) if lens else None
    return rng, tok, ki, np.ascontiguousarray(sc)


KINDS = ["normal", "equal", "zeros and ones", "few values", "one outlier", "subnormal"]
#        lengths, outer rows
SHAPES = [([1, 2, 31, 33, 159, 160, 161], 3), ([1499, 1500, 1501, 2047], 2), ([8191, 8192, 100], 60), ([8193, 9000], 80),
          ([24000, 23], 80), ([24001], 150), ([52735, 52736, 52737], 1), ([70001], 2)]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("lens,n_outer", SHAPES)
def test_topk(lens, n_outer, kind):
    budgets = [max(1, L // 3) if i % 3 != 1 else L - 1 for i, L in enumerate(lens)]
    _, tok, ki, sc = _case(kind, lens, budgets, n_outer, len(lens) + n_outer)
    sel = torch.full((n_outer, int(ki[-1]) + 2), -1, dtype=torch.int32, device=DEV)
    ties = torch.zeros((n_outer * len(lens), 4), dtype=torch.int32, device=DEV)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    B.actkv_select(torch.from_numpy(sc).to(DEV), torch.from_numpy(tok).to(DEV), int(tok[-1]),
                   torch.tensor(budgets, dtype=torch.int32, device=DEV), n_outer, len(lens), torch.from_numpy(ki).to(DEV), sel,
                   sel.shape[1], None, ties, status, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    got, tie = sel.cpu().numpy(), ties.cpu().numpy()
    for o in sorted({0, n_outer // 2, n_outer - 1}):
        for r, L in enumerate(lens):
            x = sc[o, tok[r]:tok[r + 1]]
            want = O.select_unit(x, budgets[r])
            assert np.array_equal(got[o, ki[r]:ki[r + 1]], want), (o, r)
            if len(want):
                t = np.sort(x)[::-1][len(want) - 1]
                u = o * len(lens) + r
                assert tie[u, :1].view(np.float32)[0] == t and tie[u, 3] == len(want)
                assert tie[u, 2] == (x == t).sum() and tie[u, 1] == len(want) - (x > t).sum()
    assert (got[:, ki[-1]:] == -1).all()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("lens,n_outer", [([1, 40, 1500, 1501], 2), ([8192, 700], 80), ([9000, 24000], 76), ([45568], 1)])
def test_keepscore_and_topk(lens, n_outer, kind):
    for share, prot in ((3, 0.0), (2, 0.5), (4, 0.5), (1, 0.1)):       # budget = L / share, protected prefix = prot L
        budgets = [max(1, L // share) for L in lens]
        rng, tok, ki, sc = _case(kind, lens, budgets, n_outer, 7 * len(lens) + n_outer)
        sc = np.minimum(sc, np.float32(1.0))
        protect = [int(prot * L) for L in lens]
        ks0 = (rng.random(sc.shape) ** 4).astype(np.float32)
        ks0[:, ::3] = 0.0
        d_ks = torch.from_numpy(ks0.copy()).to(DEV)
        sel = torch.full((n_outer, int(ki[-1])), -1, dtype=torch.int32, device=DEV)
        status = torch.zeros(4, dtype=torch.int32, device=DEV)
        B.actkv_keepscore_select(torch.from_numpy(sc).to(DEV), torch.from_numpy(tok).to(DEV), int(tok[-1]), max(lens), n_outer,
                                 len(lens), 0.9, 0.5, torch.tensor(protect, dtype=torch.int32, device=DEV), d_ks, None,
                                 torch.tensor(budgets, dtype=torch.int32, device=DEV), torch.from_numpy(ki).to(DEV), sel,
                                 sel.shape[1], None, None, status)
        torch.cuda.synchronize()
        assert status.cpu().tolist()[0] == 0
        got_ks, got = d_ks.cpu().numpy(), sel.cpu().numpy()
        for o in sorted({0, n_outer - 1}):
            for r, L in enumerate(lens):
                a, b = int(tok[r]), int(tok[r + 1])
                hit = O.hit_mask_unit(sc[o, a:b], 0.9)
                ks = O.keep_score_update(ks0[o, a:b], sc[o, a:b], hit, 0.5)
                assert np.array_equal(got_ks[o, a:b].view(np.uint32), ks.view(np.uint32)), (o, r)
                assert np.array_equal(got[o, ki[r]:ki[r + 1]], O.select_unit(O.rank_keys(ks, protect[r]), budgets[r])), (o, r)


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("n", [159, 160, 161, 200, 255, 256, 257, 400])
@pytest.mark.parametrize("kind", ["distinct", "equal"])
def test_keepscore_threshold_among_many_entries(kind, n, fused):
    """n entries beside one another at the threshold: n neighbouring floats in one bin, around the length of the list that is
    ranked; n equal ones, of which not all are hits."""
    rng = np.random.default_rng(n)
    L, n_outer = 700, 3
    sc = np.zeros((n_outer, L), dtype=np.float32)
    for o in range(n_outer):
        at = rng.permutation(L)
        steps = rng.permutation(n).astype(np.uint32) * (kind == "distinct")
        sc[o, at[:n]] = (np.float32(0.001).view(np.uint32) + steps).astype(np.uint32).view(np.float32)
        sc[o, at[n]] = 0.05                                # well below 90 % of the mass, and far above the others
        sc[o, at[n + 1:n + 60]] = 1e-7
    tok = torch.tensor([0, L], dtype=torch.int32, device=DEV)
    d_ks = torch.zeros((n_outer, L), device=DEV)
    mask = torch.zeros((n_outer, (L + 31) // 32), dtype=torch.int32, device=DEV)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    d_sc = torch.from_numpy(sc.copy()).to(DEV)
    if fused:
        ki = torch.tensor([0, 300], dtype=torch.int32, device=DEV)
        sel = torch.full((n_outer, 300), -1, dtype=torch.int32, device=DEV)
        B.actkv_keepscore_select(d_sc, tok, L, L, n_outer, 1, 0.9, 0.5, None, d_ks, mask,
                                 torch.tensor([300], dtype=torch.int32, device=DEV), ki, sel, 300, None, None, status)
    else:
        B.actkv_keepscore(d_sc, tok, L, n_outer, 1, 0.9, 0.5, None, d_ks, mask, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    for o in range(n_outer):
        hit = O.hit_mask_unit(sc[o], 0.9)
        assert 0 < hit.sum() < n + 1                       # the threshold lies among the n
        ks = O.keep_score_update(np.zeros(L, np.float32), sc[o], hit, 0.5)
        assert np.array_equal(d_ks.cpu().numpy()[o].view(np.uint32), ks.view(np.uint32))
        bits = np.unpackbits(mask.cpu().numpy()[o].view(np.uint8), bitorder="little")[:L].astype(bool)
        assert np.array_equal(bits, hit)
        if fused:
            assert np.array_equal(sel.cpu().numpy()[o], O.select_unit(ks, 300))


@pytest.mark.parametrize("prot", [50, 300])
@pytest.mark.parametrize("n_big", [40, 150, 400])
def test_topk_of_keep_scores_beside_the_protected_prefix(prot, n_big):
    """Keep-scores close to the largest float: the last bin of their range reaches up to +inf, as which the prefix ranks."""
    rng = np.random.default_rng(prot + n_big)
    L, budget = 2000, prot + n_big // 2
    ks0 = (1e-7 + 1e-6 * rng.random(L)).astype(np.float32)
    ks0[prot:prot + n_big] = (3.3e38 + 9e36 * rng.random(n_big)).astype(np.float32)
    d_ks = torch.from_numpy(ks0.copy()).to(DEV)
    sel = torch.full((budget,), -1, dtype=torch.int32, device=DEV)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    i32 = lambda *v: torch.tensor(v, dtype=torch.int32, device=DEV)  # noqa: E731
    B.actkv_keepscore_select(torch.full((L,), 0.25, device=DEV), i32(0, L), L, L, 1, 1, 0.0, 1.0, i32(prot), d_ks, None, i32(budget),
                             i32(0, budget), sel, budget, None, None, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    assert np.array_equal(d_ks.cpu().numpy(), ks0)         # no hits, no decay
    assert np.array_equal(sel.cpu().numpy(), O.select_unit(O.rank_keys(ks0, prot), budget))


@pytest.mark.parametrize("L,bound", [(3000, 100), (45568, 2000), (20000, 19999)])
def test_keepscore_and_topk_of_a_unit_longer_than_the_bound(L, bound):
    rng, tok, ki, sc = _case("normal", [L, 50], [L // 2, 20], 2, L)
    sc = np.minimum(sc, np.float32(1.0))
    ks0 = (rng.random(sc.shape) ** 4).astype(np.float32)
    d_ks, d_sc = torch.from_numpy(ks0.copy()).to(DEV), torch.from_numpy(sc).to(DEV)
    sel = torch.full((2, int(ki[-1])), -1, dtype=torch.int32, device=DEV)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    i32 = lambda *v: torch.tensor(v, dtype=torch.int32, device=DEV)  # noqa: E731
    B.actkv_keepscore_select(d_sc, torch.from_numpy(tok).to(DEV), int(tok[-1]), bound, 2, 2, 0.9, 0.5, i32(70, 0), d_ks, None,
                             i32(L // 2, 20), torch.from_numpy(ki).to(DEV), sel, sel.shape[1], None, None, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    assert np.array_equal(d_sc.cpu().numpy(), sc)          # left as they were
    for o in range(2):
        for r, (n, prot) in enumerate([(L // 2, 70), (20, 0)]):
            a, b = int(tok[r]), int(tok[r + 1])
            hit = O.hit_mask_unit(sc[o, a:b], 0.9)
            ks = O.keep_score_update(ks0[o, a:b], sc[o, a:b], hit, 0.5)
            assert np.array_equal(d_ks.cpu().numpy()[o, a:b].view(np.uint32), ks.view(np.uint32))
            assert np.array_equal(sel.cpu().numpy()[o, ki[r]:ki[r + 1]], O.select_unit(O.rank_keys(ks, prot), n))
