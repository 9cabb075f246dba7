"""In-place compaction at the budgets where the searches of its copy kernel take their last probe: list lengths around multiples of
33 and 33^2, lists that lie on one side of the region, random ones; both launch shapes, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2609_31395_b200 import binding as B

import parity_util as U
import test_gpu_compact_inplace as TI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [([400, 400, 400, 400], [33, 66, 264, 132]),
         ([1500, 1500, 1500], [1089, 1090, 1122]),
         ([3000, 3000, 12000], [2178, 2211, 3280]),
         ([40000], [35937])]


def _list(kind, rng, L, n):
    if kind == "below":                                    # all kept entries at the front: every search that can ends at n
        return np.arange(n)
    if kind == "above":
        return np.arange(L - n, L)
    if kind == "outside":                                  # all but a few at the front, the rest at the very end
        return np.concatenate([np.arange(n - 5), np.arange(L - 5, L)])
    return np.sort(rng.permutation(L)[:n])


@pytest.mark.parametrize("kind", ["random", "below", "above", "outside"])
@pytest.mark.parametrize("lens,budgets", CASES)
@pytest.mark.parametrize("Hkv,NL", [(1, 1), (8, 8)])       # few CTAs: 128 slots each; many: 256
def test_budgets_at_the_last_probe(lens, budgets, Hkv, NL, kind):
    if Hkv > 1 and lens[0] > 12000:
        Hkv, NL = 4, 2                                     # enough CTAs for the second launch shape all the same
    rng = np.random.default_rng(sum(budgets) + Hkv)
    inst, sel, ki, stride, max_keep = TI._direct_case(rng, lens, budgets, 16, Hkv, 64, NL)
    for o in range(NL * Hkv):
        for r, (L, n) in enumerate(zip(lens, budgets)):
            sel[o, ki[r]:ki[r + 1]] = _list(kind, rng, L, n)
    pool_before, tables_before = U.bits(inst.pool), U.oracle_tables(inst)
    d_sel = torch.from_numpy(sel).to(DEV)
    d_order = torch.full_like(d_sel, -9)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    B.actkv_compact_inplace(B.pool_desc(inst.pool), B.tables_desc(inst.page_table, inst.seq_len, inst.free_list, inst.free_count), 0,
                            NL, d_sel, stride, torch.from_numpy(ki).to(DEV), torch.tensor(budgets, dtype=torch.int32, device=DEV),
                            max_keep, d_order, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    TI._check_against_oracle(inst, pool_before, tables_before, sel, ki, budgets, d_order.cpu().numpy())
