"""Several host threads, each with a context of its own, step at the same time."""
import os
import re
import threading

import numpy as np
import pytest
import torch

from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_20332_b200", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cpp"))))
def test_no_launch_argument_is_shared(name):
    """What a launch is given (tensor maps, parameter blocks) is rebuilt from call to call: in a function-level static, two
    threads could launch with a half-written one."""
    with open(os.path.join(CSRC, name)) as f:
        found = re.findall(r"^\s+static (?:CUtensorMap|\w*Params|\w*Maps)\b.*", f.read(), re.M)
    assert not found, found


@pytest.mark.gpu
def test_two_contexts_in_two_threads():
    # query buffers of different sizes (refresh steps of 360 and 612 rows, their last block of 32 and 48, normal steps)
    jobs = [dict(P=300, G=60, A=32, B=28, R=2), dict(P=560, G=80, A=48, B=4, R=3)]
    made = []
    for i, over in enumerate(jobs):
        cfg = synth.get_config("llada8b", L=4, d=256, Hq=2, Hkv=2, dh=128, F=512, V=1000, iseed=i, **over)
        made.append((cfg, synth.make_weights(cfg, "cuda"), synth.make_prompts(cfg)))
    torch.cuda.synchronize()

    def job(cfg, w, ids):
        S = cfg["P"] + cfg["G"]
        ctx = wd.Context(cfg, w, 1, S, S, cfg["A"])
        st = wd.State(ctx, ids)
        logits = torch.zeros(cfg["A"], cfg["V"], device="cuda")
        torch.cuda.synchronize()
        st.set_taps(logits=logits)
        stream, conf = torch.cuda.Stream(), []
        for _ in range(30):
            st.step(cfg["A"], cfg["B"], cfg["R"], cfg["T"], cfg["k"], stream)
            conf.append(st.sync()["confidence"].copy())
        out = st.read(0)["ids"].copy(), np.concatenate(conf), logits.cpu().numpy()
        st.close()
        ctx.close()
        return out

    alone = [job(*m) for m in made]
    for _ in range(3):
        got = [None, None]

        def work(i):
            got[i] = job(*made[i])

        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for a, b in zip(alone, got):
            assert b is not None and all(np.array_equal(x, y) for x, y in zip(a, b))
