"""actkv_step_device refuses what the call of the stage itself refuses, before a kernel sees it."""
import pytest
import torch

from paper_2609_31395_b200 import binding as B
from paper_2609_31395_b200 import harness as H
from paper_2609_31395_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("lse_supplied", [False, True])
@pytest.mark.parametrize("field,value", [("sel_idx_dev", None), ("sel_stride", -1), ("keep_indptr_dev", None), ("score_dev", None)])
def test_selection_buffers(field, value, lse_supplied):
    wl = synth.Workload("args", 2, 2, 4, [300, 90], [20, 17], [100, 30], seed=2)
    inst = synth.generate(wl, DEV)
    comp = H.Compressor(inst.pool, inst.page_table, inst.seq_len, inst.free_list, inst.free_count, wl.n_q_heads, H.sizes_of(inst),
                        want_lse=True)
    comp.lse.fill_(6.0)
    runner = H.HostStepRunner(comp, inst.q, inst.win_indptr, inst.tok_indptr, inst.budget, wl.sm_scale, wl.causal)
    runner.stage_inputs()
    before = [t.clone() for t in (inst.page_table, inst.seq_len, inst.free_list, inst.free_count)]
    kept = getattr(runner.io, field)
    setattr(runner.io, field, value)
    with pytest.raises(B.ActKVError, match="INVALID"):
        runner.run_device(lse_supplied=lse_supplied)
    torch.cuda.synchronize()
    for t, b in zip((inst.page_table, inst.seq_len, inst.free_list, inst.free_count), before):
        assert torch.equal(t, b)
    setattr(runner.io, field, kept)
    runner.run_device(lse_supplied=lse_supplied)
    torch.cuda.synchronize()
    comp.check_status()
    assert inst.seq_len.cpu().tolist() == [100, 30]
