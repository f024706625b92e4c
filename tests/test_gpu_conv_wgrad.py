"""Accuracy of the convolutions' weight gradients (csrc/fsmi_surrogate.cu k_conv_bwd): the FP32 operands, the
layer's dz and the activations below, may lose nothing in the split into BF16 terms. Both gradients of a layer are
sums over the same dz, the bias gradient without a product, so at the step's own forward state the relative
error (2-norm, against 64 bits) of the weights' may exceed that of the biases' by the rounding of sums in FP32 at
most: 1.3 times. With two terms per operand it is 1.5 to 1.8 times."""
import numpy as np
import pytest
import torch

from oracle import surrogate as S
from paper_1905_02238_gb300 import fsmi, synth
from paper_1905_02238_gb300 import surrogate as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [128, 640])
def test_weights_as_accurate_as_biases(N):
    ratio = {2: [], 3: []}
    for seed in range(4):
        grid = synth.office_grid(300, n_obst=40, seed=11 + seed)
        poses = synth.free_cell_poses_2d(grid, 9, seed=12 + seed)
        x = fsmi.profiles_2d(*(torch.from_numpy(a).cuda() for a in (grid, poses, synth.beam_dirs_2d(72))))
        rng = np.random.default_rng(14 + seed)
        x = x[torch.from_numpy(rng.integers(0, x.shape[0], N)).cuda()].contiguous()
        th = sg.init_params(13 + seed) + rng.normal(0, 0.02, fsmi.SURR_NPARAMS).astype(np.float32)
        y = rng.normal(0.0, 1.0, N).astype(np.float32)
        params = torch.from_numpy(th).cuda()
        wb = torch.empty(fsmi.SURR_NPARAMS, dtype=torch.bfloat16, device="cuda")
        fsmi.surrogate_cast(params, wb)
        grad, loss, pred = (torch.empty(n, device="cuda") for n in (fsmi.SURR_NPARAMS, 1, N))
        ws = torch.empty(fsmi.surrogate_workspace_size(0, N), dtype=torch.uint8, device="cuda")
        fsmi.surrogate_loss_grad(params, wb, x, torch.from_numpy(y).cuda(), grad, loss, pred=pred, ws=ws)
        _, cache = S.forward(th, x.float().cpu().numpy().astype(np.float64))
        z, at = ws.view(torch.float32)[:N * 7424].cpu().numpy().astype(np.float64), 0
        for k, shape in ((1, (N, 128, 32)), (2, (N, 64, 32)), (3, (N, 32, 32)), (4, (N, 256))):
            n = int(np.prod(shape))
            cache["z%d" % k] = z[at:at + n].reshape(shape)
            cache["a%d" % k] = np.maximum(cache["z%d" % k], 0.0)
            at += n
        cache["h0"] = cache["a3"].reshape(N, -1)
        ref = S.backward(cache, S.mse(pred.cpu().numpy().astype(np.float64), y)[1])
        got, err, at = grad.cpu().numpy().astype(np.float64), {}, 0
        for name, shape in sg.LAYOUT:
            n = int(np.prod(shape))
            err[name] = np.linalg.norm(got[at:at + n] - ref[at:at + n]) / np.linalg.norm(ref[at:at + n])
            at += n
        for k in ratio:
            ratio[k].append((err["W%d" % k], err["b%d" % k]))
    for k, r in ratio.items():
        w, b = np.sqrt((np.array(r) ** 2).mean(0))
        assert w <= 1.3 * b, (k, w, b)
