"""The training step's launches overlap: two batches back to back on one workspace, eagerly and as a replayed
graph, give the bits of each alone on a fresh one, at batches around the changes of fc1's split (the tiles of
64 rows that fill two per SM: 152 SMs from 2369 and 4801 rows on)."""
import numpy as np
import pytest
import torch

from paper_1905_02238_gb300 import fsmi, synth
from paper_1905_02238_gb300 import surrogate as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M", [(1, 4096), (2368, 33), (2369, 2368), (4800, 4801), (257, 256)])
def test_back_to_back_steps(N, M):
    grid = synth.office_grid(300, n_obst=40, seed=21)
    g, p, d = (torch.from_numpy(a).cuda() for a in (grid, synth.free_cell_poses_2d(grid, 9, seed=22), synth.beam_dirs_2d(72)))
    x = fsmi.profiles_2d(g, p, d)
    th = sg.init_params(23) + np.random.default_rng(24).normal(0, 0.02, fsmi.SURR_NPARAMS).astype(np.float32)
    params = torch.from_numpy(th).cuda()
    wb = torch.empty(fsmi.SURR_NPARAMS, dtype=torch.bfloat16, device="cuda")
    fsmi.surrogate_cast(params, wb)
    batches = []
    for k, n in enumerate((N, M)):
        rows = torch.arange(n, device="cuda").mul(7 + k).remainder(x.shape[0])
        y = torch.linspace(0.0, 2.0 + k, n, device="cuda")
        out = [torch.full((m,), float("nan"), device="cuda") for m in (fsmi.SURR_NPARAMS, 1, n)]
        batches.append((x[rows].contiguous(), y, out))

    def step(b, ws):
        xb, yb, (grad, loss, pred) = b
        fsmi.surrogate_loss_grad(params, wb, xb, yb, grad, loss, pred=pred, ws=ws)

    def fresh(n):
        return torch.full((fsmi.surrogate_workspace_size(0, n),), 255, dtype=torch.uint8, device="cuda")

    want = []
    for b in batches:
        step(b, fresh(b[0].shape[0]))
        torch.cuda.synchronize()
        want.append([t.clone() for t in b[2]])
        assert all(bool(torch.isfinite(t).all()) for t in b[2])
    ws = fresh(max(N, M))

    def both():
        for b in batches:
            step(b, ws)

    def check():
        torch.cuda.synchronize()
        for b, w in zip(batches, want):
            for t, r in zip(b[2], w):
                assert torch.equal(t, r)
                t.fill_(float("nan"))

    for _ in range(3):
        both()
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        both()
    for _ in range(3):
        graph.replay()
    check()
