"""Small case for an ncu capture of the streaming expert kernels: one layer of the 30-layer workload
(hidden 2816, inter 1408, 128 experts, top-8, Q8_0), every expert resident, 64 streams, two calls."""
import sys
sys.path[:0] = [".", "tests"]
import torch, synth
from mfharness import Ctx, Shape
import paper_2607_09686_gb300 as mf
cfg = synth.CONFIGS["l30e128b64"]
T = 64
shape = Shape(1, cfg.hidden, cfg.n_experts, cfg.top_k, cfg.inter, cfg.qtype)
ctx = Ctx(shape, cfg.n_experts, max_tokens=T, workers=16)
r = synth.routes(0, 0, 0, cfg.n_experts, cfg.top_k, T, 1.0, 0.0)
x = torch.from_numpy(synth.activations(0, 0, 0, 0, T, cfg.hidden)).cuda()
b = torch.from_numpy(synth.plant_bias(r, cfg.n_experts)).cuda()
y = torch.empty(T, cfg.hidden, device="cuda")
for rep in range(2):
    mf.mf_moe_forward(ctx.h, 0, x, ctx.wr[0], b, T, y)
torch.cuda.synchronize()
assert mf.mf_check(ctx.h) == 0
print("ok")
ctx.close()
