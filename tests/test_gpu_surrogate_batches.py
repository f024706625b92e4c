"""The surrogate's training step and inference at the edges of their tiles: batches around the strips
of 16, the head's blocks of 32 rows, fc1's tiles of 128 rows and its splits of the batch, and a warp's
queue grabs; weights off a 16-byte boundary. The training step against the FP64 oracle at the step's own
forward state, with the bounds of test_gpu_surrogate.py."""
import numpy as np
import pytest
import torch

from oracle import surrogate as S
from paper_1905_02238_gb300 import fsmi, synth
from paper_1905_02238_gb300 import surrogate as sg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    grid = synth.office_grid(300, n_obst=40, seed=11)
    poses = synth.free_cell_poses_2d(grid, 9, seed=12)
    g, p, d = (torch.from_numpy(a).cuda() for a in (grid, poses, synth.beam_dirs_2d(72)))
    x = fsmi.profiles_2d(g, p, d)
    th = sg.init_params(13) + np.random.default_rng(14).normal(0, 0.02, fsmi.SURR_NPARAMS).astype(np.float32)
    params = torch.from_numpy(th).cuda()
    wb = torch.empty(fsmi.SURR_NPARAMS, dtype=torch.bfloat16, device="cuda")
    fsmi.surrogate_cast(params, wb)
    return g, p, d, x, th, params, wb


def _step(params, wb, x, y):
    N = x.shape[0]
    grad, loss, pred = (torch.full((n,), float("nan"), device="cuda") for n in (fsmi.SURR_NPARAMS, 1, N))
    ws = torch.full((fsmi.surrogate_workspace_size(0, N),), 255, dtype=torch.uint8, device="cuda")
    fsmi.surrogate_loss_grad(params, wb, x, y, grad, loss, pred=pred, ws=ws)
    return grad, loss, pred, ws


@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 127, 128, 129, 256, 257, 513])
def test_training_step(case, N):
    _, _, _, x, th, params, wb = case
    x = x[:N].contiguous()
    y = np.random.default_rng(N).uniform(0, 3, N).astype(np.float32)
    grad, loss, pred, ws = _step(params, wb, x, torch.from_numpy(y).cuda())
    rpred, cache = S.forward(th, x.float().cpu().numpy().astype(np.float64))
    np.testing.assert_allclose(pred.cpu().numpy(), rpred, rtol=2e-5, atol=2e-5 * np.abs(rpred).max())
    zf, at = ws.view(torch.float32)[:N * 7424].cpu().numpy().astype(np.float64), 0
    for k, shape in (("z1", (N, 128, 32)), ("z2", (N, 64, 32)), ("z3", (N, 32, 32)), ("z4", (N, 256))):
        n = int(np.prod(shape))
        cache[k] = zf[at:at + n].reshape(shape)
        at += n
    cache["a1"], cache["a2"], cache["a3"], cache["a4"] = (np.maximum(cache[k], 0.0) for k in ("z1", "z2", "z3", "z4"))
    cache["h0"] = cache["a3"].reshape(N, -1)
    rloss, dpred = S.mse(pred.cpu().numpy().astype(np.float64), y)
    assert abs(float(loss.item()) - rloss) <= 5e-5 * rloss
    rgrad = S.backward(cache, dpred)
    acache = dict(cache)
    acache["p"] = {k: np.abs(v) for k, v in cache["p"].items()}
    for k in ("a0", "a1", "a2", "a3", "a4", "h0"):
        acache[k] = np.abs(cache[k])
    bound = S.backward(acache, np.abs(dpred))
    assert np.all(np.abs(grad.cpu().numpy().astype(np.float64) - rgrad) <= 2e-4 * bound + 1e-12)


def test_weights_off_a_16_byte_boundary(case):
    _, _, _, x, _, params, wb = case
    x = x[:65].contiguous()
    y = torch.linspace(0.0, 2.0, 65, device="cuda")
    off = torch.empty(fsmi.SURR_NPARAMS + 1, dtype=torch.bfloat16, device="cuda")[1:]
    off.copy_(wb)
    assert off.data_ptr() % 16 != 0
    for a, b in zip(_step(params, wb, x, y)[:3], _step(params, off, x, y)[:3]):
        assert torch.equal(a, b)


def test_predict_batches(case):
    g, p, d, x, th, params, wb = case
    full = fsmi.surrogate_predict(params, wb, grid=g, poses=p, dirs=d)
    assert torch.equal(full, fsmi.surrogate_predict(params, wb, x=x))
    ref, _ = S.forward(th, x.float().cpu().numpy().astype(np.float64), act_bf16=True)
    assert np.abs(full.cpu().numpy() - ref).max() <= 1e-3 * max(1.0, np.abs(ref).max())
    for n in (1, 3, 4, 5, 31, 33, 127, 128, 129, 600):
        assert torch.equal(fsmi.surrogate_predict(params, wb, x=x[:n].contiguous()), full[:n])
    assert fsmi.device_status() == 0
