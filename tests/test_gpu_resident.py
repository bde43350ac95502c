"""AUTO on FP32 grids up to 384 columns wide (one cluster holds the state, one launch a stretch of
steps) against the one-thread-per-cell kernel: the same bits, at the edges of every lane width (2, 4,
8 and 12 columns a lane, with a last lane that overlaps the one before it), with 1 to 4 rows a warp, one
to sixteen blocks, and on both sides of the range's ends."""
import pytest
import torch

import rdcnn_inputs as inp
from _util import gpu_run

pytestmark = pytest.mark.gpu

SHAPES = [(1, 16), (1, 64), (2, 17), (5, 96), (15, 15), (16, 16), (17, 63), (31, 65), (33, 33), (40, 200), (61, 130),
          (64, 64), (100, 128), (129, 127), (200, 250), (255, 251), (256, 256), (260, 255), (512, 256), (513, 256),
          (1023, 49), (1024, 100), (1025, 64), (1, 257), (17, 268), (48, 257),
          (90, 383), (64, 384), (256, 260), (256, 384), (257, 300), (40, 385)]
MODELS = [("periodic", "fhn"), ("zeroflux", "fhn"), ("periodic", "cenn"), ("zeroflux", "cenn"), ("zeroflux", "none")]


def _gene(reaction):
    return {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0} if reaction == "cenn" \
        else inp.default_params()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("boundary,reaction", MODELS)
def test_auto_matches_generic_bitwise(rd, shape, boundary, reaction):
    x, y = inp.uniform_field(41, *shape), 0.7 * inp.uniform_field(42, *shape)
    for T in (1, 2, 3, 30):
        a, b = (gpu_run(rd, x, y, _gene(reaction), T, torch.float32, v, reaction=reaction, boundary=boundary)
                for v in ("auto", "generic"))
        assert (a[0] == b[0]).all() and (a[1] == b[1]).all(), T


@pytest.mark.parametrize("shape", [(64, 64), (37, 121), (256, 256)])
def test_planes_off_their_alignment_and_captured_runs(rd, shape):
    """Planes one element past an aligned address, run eagerly and from the caller's captured graph."""
    nn, nm = shape
    base = [torch.zeros(nn * nm + 2, device="cuda") for _ in range(2)]
    u, v = (t[1:1 + nn * nm].view(nn, nm) for t in base)
    x = torch.from_numpy(inp.uniform_field(43, nn, nm)).float().cuda()
    u.copy_(x), v.copy_(-x)
    rd.run(u, v, inp.default_params(), 25, variant="auto")
    assert all(float(t[0]) == 0.0 and float(t[-1]) == 0.0 for t in base)
    g = rd.Grid(nn, nm, inp.default_params())
    g.set_state(x, -x).run(25)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        c = rd.Grid(nn, nm, inp.default_params())
        c.set_state(x, -x)
        with torch.cuda.graph(graph, stream=side):
            c.run(5)
        for _ in range(5):
            graph.replay()
    torch.cuda.synchronize()
    ref = gpu_run(rd, x.double().cpu().numpy(), -x.double().cpu().numpy(), inp.default_params(), 25, torch.float32, "generic")
    for got in ((u, v), (g.u, g.v), (c.u, c.v)):
        assert all((t.cpu().numpy() == r).all() for t, r in zip(got, ref))


@pytest.mark.parametrize("boundary,reaction", MODELS)
@pytest.mark.parametrize("shape", [(2, 17), (16, 16), (64, 64), (61, 130), (256, 256), (256, 384), (1024, 100)])
def test_a_wait_that_gives_up_leaves_no_cell_that_looks_like_a_result(rd, shape, boundary, reaction):
    """Every wait runs out in the first step (an arrival that nobody makes): the launch ends, both planes
    are NaN in every cell, and the next run on the same planes gives its bits as ever."""
    from paper_2102_10340_gb300 import _lib as L

    x, y = (torch.from_numpy(inp.uniform_field(s, *shape)).float().cuda() for s in (44, 45))
    g = rd.Grid(*shape, _gene(reaction), reaction=reaction, boundary=boundary)
    g.set_state(x, y)
    rc = g.lib.rdcnn_run_cluster(g.h, 9, 1)
    if rc == L.EINVAL and "no room" in L.last_error():
        pytest.skip("this device runs no cluster of 16 blocks")
    L.check(rc)
    torch.cuda.synchronize()
    assert torch.isnan(g.u).all() and torch.isnan(g.v).all()
    out = []
    for run in (lambda: L.check(g.lib.rdcnn_run_cluster(g.h, 9, 0)), lambda: g.run(9, variant="generic")):
        g.set_state(x, y)
        run()
        out.append(g.state())
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_a_tuned_grid_still_runs_in_one_launch(rd):
    """The tuner finds the cluster launch of a small FP32 grid and leaves it in force."""
    from paper_2102_10340_gb300 import autotune

    g = rd.Grid(64, 64, inp.default_params())
    best = autotune.tune_grid(g, torch.from_numpy(inp.uniform_field(46, 64, 64)).float().cuda(), force=True)
    before = rd.launch_count()
    g.run(500, variant=best["variant"], k=best["k"])
    assert best["variant"] == "auto" and rd.launch_count() - before == 1


def test_cluster_runs_are_refused_where_the_grid_does_not_fit(rd):
    from paper_2102_10340_gb300 import _lib as L

    for shape, dtype in (((64, 15), torch.float32), ((64, 385), torch.float32), ((257, 300), torch.float32),
                         ((64, 64), torch.float64)):
        g = rd.Grid(*shape, inp.default_params(), dtype=dtype)
        assert g.lib.rdcnn_run_cluster(g.h, 1, 0) == L.EINVAL and "fit" in L.last_error()
    g = rd.Grid(64, 64, inp.default_params())
    assert g.lib.rdcnn_run_cluster(g.h, -1, 0) == L.EINVAL


def test_runs_on_two_streams_at_once(rd):
    """Clusters of two grids on two streams, many short runs each: each grid gets its own bits."""
    out = []
    for parallel in (True, False):
        grids = []
        for i in range(4):
            s = torch.cuda.Stream() if parallel else torch.cuda.current_stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s):
                g = rd.Grid(64 + 50 * i, 80, inp.default_params())
                g.init(torch.from_numpy(inp.uniform_field(50 + i, g.nn, g.nm)).float().cuda())
            grids.append((g, s))
        for _ in range(12):
            for g, s in grids:
                with torch.cuda.stream(s):
                    g.run(17)
        torch.cuda.synchronize()
        out.append([(g.u.clone(), g.v.clone()) for g, _ in grids])
    for a, b in zip(*out):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
