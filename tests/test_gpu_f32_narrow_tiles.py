"""fp32 projections in tiles of up to 64 columns, more of them than SMs (two blocks to an SM): d_head 20, 40 and 64 (weight boxes of
32, 48 and 64 rows), contractions of one chunk of two steps, of three and of seventeen, lists whose last tiles are short, dAhat over as
many tiles; d_head 132, 150 and 192 in three tiles (boxes of 48 and 64 rows, the last tile 4 columns past a box of 16, 22, and whole),
output and dx of the values in tiles of 64 columns over five and six steps, the last one 4 positions long, 22, and whole."""
import numpy as np
import pytest
import torch

from oracle.switchhead_backward import switchhead_backward
from oracle.switchhead_oracle import switchhead_forward
from paper_2312_07987_b200 import binding, inputs

pytestmark = pytest.mark.gpu
# max-abs error / largest value: an fp32 sum of K products differs from the fp64 one by about sqrt(K) 2^-24 of its own
# size, times 5 for the largest of ~1e5 values: K <= 2400 tokens, 1.5e-5
TOL = 1.5e-5


@pytest.mark.parametrize("B,T,M,H,D,E,k", [
    (16, 130, 64, 8, 20, 3, 2),
    (13, 97, 1088, 6, 64, 4, 1),
    (8, 300, 192, 3, 40, 5, 3),
    (24, 100, 192, 2, 132, 4, 2),
    (10, 130, 448, 3, 150, 5, 3),
    (30, 81, 256, 2, 192, 3, 2),
])
def test_f32_narrow_tiles(B, T, M, H, D, E, k):
    cfg = inputs.LayerConfig("narrow", inputs.DTYPE_F32, B, T, M, H, D, E, k, seed=T + M)
    lists = H * (B * T * k // 128 + E // 2)
    tiles = -(-B * T // 128) * 2 * H + lists
    if D > 128:
        tiles = min(2 * tiles, lists * -(-M // 128))
    assert tiles > torch.cuda.get_device_properties(0).multi_processor_count
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
