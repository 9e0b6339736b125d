"""A refresh step without block taps computes the last block for the active rows only: same logits, same cache."""
import pytest
import torch

from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth
from wd_harness import Parity

pytestmark = pytest.mark.gpu
DEV = "cuda"


# the smallest row count that takes it (257), grouped-query heads and several sequences (one of them shorter), more active
# rows than a query tile, exactly half of the rows active, one active row; 2 * active > rows (does not take it)
@pytest.mark.parametrize("Hq,Hkv,batch,P,G,A,B", [(2, 2, 1, 217, 100, 30, 10), (4, 1, 3, 150, 90, 16, 20), (2, 2, 2, 300, 300, 140, 60),
                                                  (2, 2, 1, 130, 200, 160, 30), (4, 2, 1, 260, 60, 1, 10), (2, 2, 1, 100, 300, 200, 60)])
def test_active_rows_of_the_last_block(Hq, Hkv, batch, P, G, A, B):
    cfg = synth.get_config("llada8b", L=2, d=256, Hq=Hq, Hkv=Hkv, dh=128, F=512, V=1000, P=P, G=G)
    w = synth.make_weights(cfg, DEV)
    ids = synth.make_prompts(cfg, batch=batch)
    if batch > 1:
        ids[1, P - 40:] = cfg["mask_id"]                # a shorter prompt
    S = P + G
    runs, launches = [], []
    for all_taps in (True, False):
        ctx = wd.Context(cfg, w, batch, S, batch * S, batch * A)
        st = wd.State(ctx, ids)
        logits = torch.zeros(batch * A, cfg["V"], device=DEV)
        taps = dict(layer_out=torch.zeros(2 * batch * S * 256, device=DEV)) if all_taps else {}
        st.set_taps(logits=logits, **taps)
        out = []
        for _ in range(2):                              # a refresh, then a normal step that reads the cache it wrote
            _, info = st.step(A, B, 8, 2, 0)            # k = 0: nothing is unmasked, both runs keep the same state
            st.sync()
            out.append(logits[:info["n_active"]].clone())
            launches.append((info["n_rows"], info["n_launches"]))
        runs.append(out)
        st.close()
        ctx.close()
    rows = launches[0][0]
    assert rows > 256
    took = 2 * batch * A <= rows
    # per block: keys/values, gather, queries and two rotations instead of one of each; no residual kernels for the tap
    assert (launches[2][1] == launches[0][1] + 1) == took
    for full, act in zip(*runs):
        # the same bf16 pipeline with other splits of the sums: bounded by the tolerance of a block's output
        assert float((full - act).norm() / full.norm()) < 1e-2


# grouped-query heads and three sequences, one of them shorter; full heads, more active rows than a query tile and fewer than half
@pytest.mark.parametrize("Hq,Hkv,batch,P,G,A,B", [(4, 1, 3, 150, 90, 16, 20), (2, 2, 2, 300, 300, 140, 60)])
def test_untapped_blocks_against_the_oracle(Hq, Hkv, batch, P, G, A, B):
    """The path that steps take in use: only the logits are tapped.  Index sets, logits, chosen tokens of a refresh step, of the
    two normal steps that read the cache it wrote, and of the next refresh."""
    cfg = synth.get_config("llada8b", L=2, d=256, Hq=Hq, Hkv=Hkv, dh=128, F=512, V=1000, P=P, G=G)
    w = synth.make_weights(cfg, DEV, gain_jitter=0.1)
    ids = synth.make_prompts(cfg, batch=batch)
    ids[1, P - 40:] = cfg["mask_id"]
    par = Parity(cfg, w, ids, block_taps=False)
    for i in range(4):
        info = par.step(A, B, 3, 2, 1)["info"]
        assert info["is_refresh"] == (i % 3 == 0)
        if info["is_refresh"]:
            assert info["n_rows"] > 256 and 2 * info["n_active"] <= info["n_rows"]
    par.check_state_mirror()
    par.close()
