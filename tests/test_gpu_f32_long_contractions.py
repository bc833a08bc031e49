"""fp32 layer: contractions of more than 1024 positions (the small products' accumulator is read back more than once), at
that boundary and one step past it, over d_model and over an expert's tokens, with as many tiles as leave none of them
split; and column tiles of 112 and of two times 80 columns."""
import numpy as np
import pytest
import torch

from oracle.switchhead_backward import switchhead_backward
from oracle.switchhead_oracle import switchhead_forward
from paper_2312_07987_b200 import binding, inputs

pytestmark = pytest.mark.gpu
# max-abs error / largest value: an fp32 sum of K products differs from the fp64 one by about sqrt(K) 2^-24 of its own
# size, times 5 for the largest of ~1e5 values: K <= 2112, 1.4e-5
TOL = 1.4e-5


@pytest.mark.parametrize("T,M,H,D,E,k", [
    (130, 1024, 1, 112, 2, 1),       # 32 steps: the last one ends the period
    (70, 1088, 2, 112, 3, 2),        # 34 steps
    (65, 2112, 1, 140, 2, 2),        # 66 steps; two column tiles a head
    (1060, 1024, 4, 40, 1, 1),       # 34 steps over the tokens: 72 + 64 tiles of weight gradients, none split
])
def test_f32_long_contractions(T, M, H, D, E, k):
    cfg = inputs.LayerConfig("long", inputs.DTYPE_F32, 1, T, M, H, D, E, k, seed=T + M)
    inp = inputs.make_inputs(cfg)
    G = np.random.default_rng(5).standard_normal(inp.x.shape).astype(np.float32)
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, cfg.dtype)
    y = layer.sh_forward(x)
    got = dict(layer.sh_backward(x, torch.from_numpy(G).cuda()), y=y)
    torch.cuda.synchronize()
    assert layer.sh_last_status() == 0
    layer.sh_check_guards()
    args = (inp.x, inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, cfg.k)
    want = dict(switchhead_backward(*args, G, inp.bias_s, inp.bias_d))
    want["y"] = switchhead_forward(*args, inp.bias_s, inp.bias_d, return_stages=False)["y"]
    for name in ("y", "dx", "dWq", "dWk", "dWv", "dWo", "dWs", "dWd"):
        r = want[name]
        a = got[name].cpu().numpy().astype(np.float64).reshape(r.shape)
        assert np.abs(a - r).max() / (np.abs(r).max() or 1.0) < TOL, name
    layer.close()
