"""The inference front end on frames that start on 16 bytes and on frames that do not: the same actions."""
import pytest
import torch

from paper_2602_21203_gb300 import synth

pytestmark = pytest.mark.gpu


# factor, squinted size: whole and part blocks of chunks, rows of one chunk and of many, widths that are no multiple of 16
@pytest.mark.parametrize("f,h,w", [(4, 16, 16), (4, 32, 32), (4, 24, 20), (2, 16, 24), (2, 17, 40), (1, 32, 32), (1, 20, 48),
                                   (1, 18, 18), (2, 15, 15), (4, 13, 13)])
@pytest.mark.parametrize("rows", [1, 37])
def test_act_frames_aligned_or_not(f, h, w, rows):
    from paper_2602_21203_gb300 import lib
    cfg = synth.make_config("small_b32", obs_h=f * h, obs_w=f * w, squint_f=f, shift_pad=0)
    learner = lib.Learner(cfg, None)
    obs, prop = synth.make_obs_batch(rows, cfg, 3, device="cuda")
    outs = []
    for off in (0, 5, 16):
        buf = torch.empty(obs.numel() + off, dtype=torch.uint8, device="cuda")
        buf[off:] = obs.reshape(-1)
        out = torch.empty(rows, cfg["action_dim"], device="cuda")
        learner.act([lib.Learner.request(buf[off:], prop, out, key=1, sample=False)])
        torch.cuda.synchronize()
        outs.append(out)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    assert bool(torch.isfinite(outs[0]).all())
    learner.close()
