"""The one-launch encoder forward against the layer-by-layer tensor-core convolutions: the same bits."""
import numpy as np
import pytest
import torch

from paper_2602_21203_gb300 import synth
from util import ring_to_device, split_params

pytestmark = pytest.mark.gpu


# squinted h, w, layers, batch: one to three tiles of the first layer, last rows of a tile, odd and uneven sizes,
# two to five layers, fewer images than SMs, a round and a bit, an input whose bytes are no multiple of 16 (the
# layer-by-layer path) and the training shape
@pytest.mark.parametrize("h,w,layers,batch", [(32, 32, 4, 37), (32, 32, 4, 512), (12, 12, 2, 1), (16, 16, 3, 5), (24, 40, 4, 80),
                                              (40, 38, 3, 150), (32, 32, 5, 9), (34, 30, 2, 305), (28, 22, 4, 64),
                                              (17, 23, 3, 6)])
def test_encoder_equals_the_layers(h, w, layers, batch):
    from paper_2602_21203_gb300 import lib, ops
    cfg = synth.make_config("train_b512", ring_size=64, obs_h=2 * h, obs_w=2 * w, squint_f=2, shift_pad=2, batch=batch,
                            conv_layers=layers, proj_dim=32, hidden=[64, 64], atoms=11)
    learner = lib.Learner(cfg, ring_to_device(synth.make_ring(cfg, 0)), precision=lib.PREC_BF16)
    P = split_params(learner.params(), cfg)
    learner.update(1)
    x = torch.from_numpy(learner.debug("x_t").reshape(batch, 3, h, w)).cuda()
    z = learner.debug("z_t")
    dev = lambda name: torch.from_numpy(P[name].astype(np.float32)).cuda()
    convs = [(dev(f"enc.conv{i}.w"), dev(f"enc.conv{i}.b")) for i in range(layers)]
    y, hh, ww = ops.conv0_bf16(x, *convs[0], 2), (h - 3) // 2 + 1, (w - 3) // 2 + 1
    for wt, b in convs[1:]:
        y, chw = ops.conv32_fwd(y, hh, ww, ops.conv32_layouts(wt)[0], b)
        hh, ww = hh - 2, ww - 2
    assert np.array_equal(z.reshape(-1), chw.cpu().numpy().reshape(-1))
    # inference reads the same encoder: a row alone and inside a ragged batch of two rounds give the same action
    learner.refresh_policy()
    obs, prop = synth.make_obs_batch(700, cfg, 3, device="cuda")
    out = torch.empty(700, cfg["action_dim"], device="cuda")
    one = torch.empty(1, cfg["action_dim"], device="cuda")
    learner.act([lib.Learner.request(obs, prop, out, key=1, sample=False)])
    learner.act([lib.Learner.request(obs[699:], prop[699:], one, key=1, sample=False)])
    torch.cuda.synchronize()
    assert torch.equal(out[699:], one)
    learner.close()
