"""Range classes of a mixed call whose launches overlap: two different streams of sets back to back on one
workspace, eagerly and as one replayed graph, equal the call without a plan (one launch) bit for bit. A class may
be missing, hold one ray, or hold the bulk of the work, and the plan may have to be given up."""
import numpy as np
import pytest
import torch

from paper_1905_02238_gb300 import fsmi, synth

pytestmark = pytest.mark.gpu

BULK = [(fsmi.SET_2D, 0, 24, 0, 90, 30.0), (fsmi.SET_3D, 0, 6, 0, 120, 90.0, 0), (fsmi.SET_2D, 3, 20, 0, 90, 310.0),
        (fsmi.SET_3D, 1, 5, 0, 120, 15.0, 0)]
EDGES = [(fsmi.SET_3D, 2, 1, 5, 1, 300.0, 0), (fsmi.SET_2D, 7, 1, 0, 1, 16.0), (fsmi.SET_2D, 7, 1, 0, 90, 400.0),
         (fsmi.SET_3D, 0, 1, 0, 3, 64.0, 0), (fsmi.SET_2D, 1, 0, 0, 90, 100.0), (fsmi.SET_2D, 2, 2, 0, 90, 65.0)]


@pytest.mark.parametrize("first,second", [(BULK, EDGES), (EDGES, BULK), (BULK[::-1], BULK[:1]), (EDGES[:1], BULK)])
@pytest.mark.parametrize("bad_plan", [False, True])
def test_overlapping_classes(first, second, bad_plan):
    grid = synth.office_grid(512, n_obst=60, seed=51)
    vol = synth.voxel_world(96, 80, 48, n_boxes=16, seed=52, noise_seed=53, noise_frac=0.05)
    cuda = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (
        grid, synth.free_cell_poses_2d(grid, 24, seed=54), synth.beam_dirs_2d(90), vol,
        synth.free_voxel_poses(vol, 6, seed=55, zlo=6, zhi=40), synth.pinhole_dirs(12, 10, 100.0))]
    g, p2, d2, v, p3, d3 = cuda
    b = dict(variant=fsmi.EXACT, sigma=2.0, delta_occ=1.5, delta_emp=0.67, max_range=400.0)
    kw = dict(grid=g, poses2=p2, dirs2=d2, prm2=fsmi.Params(**b), volumes=fsmi.make_volumes([v], "cuda"), poses3=p3,
              dirs3=d3, prm3=fsmi.Params(**dict(b, run_cap=64)))
    calls = []
    for sets in (first, second):
        # a kind that does not exist, on an empty set: no item changes, but no plan takes it
        st, n = fsmi.make_sets(sets + [(7, 0, 0, 0, 90, 10.0)] * bad_plan, "cuda")
        calls.append((st, n, torch.zeros(n, device="cuda")))
    nb = max(fsmi.mixed_workspace_size(g.numel(), c[0].shape[0]) for c in calls)
    ws = torch.full((nb,), 0xA5, dtype=torch.uint8, device="cuda")
    small = torch.empty(fsmi.workspace_size(fsmi.FN_EVAL_2D, g.numel()), dtype=torch.uint8, device="cuda")
    want = [fsmi.eval_mixed(*fsmi.make_sets(s, "cuda"), ws=small, **kw) for s in (first, second)]

    def run():
        for st, n, out in calls:
            fsmi.eval_mixed(st, n, out=out, ws=ws, **kw)

    def check():
        torch.cuda.synchronize()
        for (_, _, out), w in zip(calls, want):
            assert torch.equal(out.view(torch.int32), w.view(torch.int32))
            out.fill_(float("nan"))

    for _ in range(3):
        run()
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for _ in range(3):
        graph.replay()
    check()
