"""With less memory free than the size queries ask for, the binding takes a smaller workspace: the
evaluation, the DMC step and the batch run as they do on a smaller workspace of the caller's."""
import pytest
import torch

from synth import config_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


def test_eval_dmc_batch_with_little_memory():
    from paper_1209_6630_gb300 import QmcBatch, QmcSystem
    s = config_system("434e")
    R = torch.from_numpy(make_walkers(s, 37, first=99000)).to(dev)
    q = QmcSystem(s, 0)
    need = q.workspace_size(37, "mixed")
    ref = {k: v.clone() for k, v in q.eval(R, precision="mixed").items()}
    q._ws.clear()
    a, b = q.walker_state(37), q.walker_state(37)
    for k in ("drift", "e_loc", "logpsi", "sign", "status"):
        a[k].copy_(ref[k])
    a["R"].copy_(R)
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(dev).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + 0.8 * need) / total)
    try:
        out = q.eval(R, precision="mixed")
        ws = q.workspace(37, "mixed")
        assert ws.numel() < need and q.workspace(37, "mixed") is ws
        assert torch.equal(out["status"], ref["status"])
        assert (out["logpsi"] - ref["logpsi"]).abs().max().item() < 1e-6
        del ws
        q._ws.clear()
        q.dmc_step(a, b, tau=1e-4, e_trial=-500.0, seed=3, step=1, precision="mixed")
        assert torch.isfinite(b["logpsi"]).all()
        q._ws.clear()
        batch = QmcBatch([(q, R)], precision="mixed", graph=False)
        assert (batch.eval()[0]["logpsi"] - ref["logpsi"]).abs().max().item() < 1e-6
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
