"""Plans of one context on several streams: one whose stream is held up must not hold up the others (the batched form plans on
four streams), nor any number of them a plan on a high-priority stream. A sleep kernel of bounded length holds the
first stream up; the others' plans have to be done, and right, while it still runs. In a process of its own, with
a hardware queue for every stream (streams that share one wait for each other)."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 20_001  # above the single-launch size, so that the plan has two halves


def check():
    from oracle import oracle as O
    from paper_2607_14513_gb300 import gsc
    from paper_2607_14513_gb300 import synthetic as S
    ctx = gsc.Context(0)
    sc = S.make_scene(N, 8)
    pos, sh = torch.from_numpy(sc.pos).cuda(), torch.from_numpy(sc.sh).cuda()
    want = O.scales(sc.sh)
    perm = O.plan(sc.pos, O.quantise(sc.sh, want), 4096, 1)
    high = torch.cuda.Stream(priority=-1)
    for held_plans, others in ((1, [torch.cuda.Stream() for _ in range(3)]), (4, [high])):
        ws = [ctx.workspace(N) for _ in range(held_plans + len(others))]
        for w in ws:                       # once each, outside the measurement
            gsc.gsc_plan_reorder(ctx, pos, sh, ws=w)
        torch.cuda.synchronize()
        held, end = torch.cuda.Stream(), torch.cuda.Event()
        with torch.cuda.stream(held):
            torch.cuda._sleep(4_000_000_000)   # about 2 s
        late = [gsc.gsc_plan_reorder(ctx, pos, sh, ws=w, stream=held) for w in ws[:held_plans]]
        end.record(held)
        got = [gsc.gsc_plan_reorder(ctx, pos, sh, ws=w, stream=s) for w, s in zip(ws[held_plans:], others)]
        for s in others:
            s.synchronize()
        assert not end.query()
        torch.cuda.synchronize()
        for p, s in got + late:
            assert np.array_equal(s.cpu().numpy(), want) and np.array_equal(p.cpu().numpy(), perm)
    ctx.close()


def test_plans_do_not_wait_for_a_held_stream():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=root, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CUDA_DEVICE_MAX_CONNECTIONS="32", PYTHONPATH=root))
    assert r.returncode == 0, r.stdout + r.stderr


if __name__ == "__main__":
    check()
