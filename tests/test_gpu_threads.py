"""Two threads, each with its own system, stream and workspace, one of the systems with a Jastrow factor and one
larger than the other: every call runs and gives what it gives alone."""
import threading

import pytest
import torch

from synth import config_system, make_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_two_threads(precision):
    from paper_1209_6630_gb300 import QmcSystem
    parts = []
    for i, s in enumerate((make_system(9, 3, 3, 20, seed=21), config_system("158e"), make_system(9, 3, 3, 20, seed=21))):
        q = QmcSystem(s, 0)
        if i == 2:
            q.set_jastrow(dict(a_par=0.25, a_anti=0.5, b_ee=1.0, a_en=0.8, b_en=2.0))
        R = torch.from_numpy(make_walkers(s, 2, first=94000)).to(dev)
        parts.append((q, R, {k: v.clone() for k, v in q.eval(R, precision=precision).items()}))
    torch.cuda.synchronize()
    errors = []

    def work(q, R, ref):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            out, ws = q.alloc_out(2), q.workspace(2, precision)
            try:
                for _ in range(300):
                    q.eval(R, precision=precision, out=out, ws=ws)
                stream.synchronize()
                assert all(torch.equal(out[k], ref[k]) for k in ("logpsi", "drift", "e_loc", "status"))
            except Exception as e:                        # noqa: BLE001
                errors.append(repr(e))

    ts = [threading.Thread(target=work, args=p) for p in parts]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
