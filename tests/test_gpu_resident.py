"""FP32 grids up to 384 columns wide held by one cluster (rdcnn_run_cluster, and AUTO where it is the
faster way) against the one-thread-per-cell kernel: the same bits, at the edges of every lane width (2, 4,
8 and 12 columns a lane, with a last lane that overlaps the one before it), with 1 to 4 rows a warp, one
to sixteen blocks; and which launches AUTO takes, on both sides of the range's ends."""
import pytest
import torch

import rdcnn_inputs as inp
from _util import gpu_run

pytestmark = pytest.mark.gpu

SHAPES = [(1, 16), (1, 64), (2, 17), (5, 96), (15, 15), (16, 16), (17, 63), (31, 65), (33, 33), (40, 200), (61, 130),
          (64, 64), (100, 128), (129, 127), (200, 250), (255, 251), (256, 256), (260, 255), (512, 256), (513, 256),
          (1023, 49), (1024, 100), (1025, 64), (1, 257), (17, 268), (48, 257),
          (90, 383), (64, 384), (256, 260), (256, 384), (257, 300), (40, 385)]
OUTSIDE = [(15, 15), (513, 256), (1025, 64), (257, 300), (40, 385)]  # SHAPES that no cluster holds
MODELS = [("periodic", "fhn"), ("zeroflux", "fhn"), ("periodic", "cenn"), ("zeroflux", "cenn"), ("zeroflux", "none")]


def _gene(reaction):
    return {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0} if reaction == "cenn" \
        else inp.default_params()


def _cluster(g, T, give_up=0):
    """T steps by cluster launches; skips on a device that has no room for sixteen blocks."""
    from paper_2102_10340_gb300 import _lib as L

    rc = g.lib.rdcnn_run_cluster(g.h, T, give_up)
    if rc == L.EINVAL and "no room" in L.last_error():
        pytest.skip("this device runs no cluster of 16 blocks")
    L.check(rc)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("boundary,reaction", MODELS)
def test_cluster_and_auto_match_generic_bitwise(rd, shape, boundary, reaction):
    x, y = (torch.from_numpy(s * inp.uniform_field(i, *shape)).float().cuda() for i, s in ((41, 1.0), (42, 0.7)))
    for T in (1, 2, 3, 30, 150):
        out = []
        for how in ("generic", "auto", "cluster"):
            g = rd.Grid(*shape, _gene(reaction), reaction=reaction, boundary=boundary)
            g.set_state(x, y)
            before = rd.launch_count()
            if how != "cluster":
                g.run(T, variant=how)
            elif shape not in OUTSIDE:
                _cluster(g, T)
                assert rd.launch_count() - before == 1
            else:
                continue
            out.append(g.state())
        assert all(torch.equal(a, b) for o in out[1:] for a, b in zip(o, out[0])), T


@pytest.mark.parametrize("shape,T,launches", [((1, 16), 30, 1), ((64, 64), 1, 1), ((64, 64), 30, 1), ((64, 15), 30, None),
                                              ((1024, 64), 30, 1), ((1025, 64), 30, None), ((512, 256), 8, 2),
                                              ((512, 256), 300, 1), ((513, 256), 300, None), ((256, 384), 100, 1),
                                              ((257, 384), 100, None), ((256, 385), 100, None), ((400, 256), 6, 2),
                                              ((251, 253), 30, 1), ((64, 64), 8192 + 3, 2)])
def test_which_launches_auto_takes(rd, shape, T, launches):
    """One launch (of at most 8192 steps) for a whole run in the cluster's range, more than one outside it
    and for short runs of its largest grids; the same state as in calls of 101 steps."""
    x = torch.from_numpy(inp.uniform_field(47, *shape)).float().cuda()
    g, h = (rd.Grid(*shape, inp.default_params()) for _ in range(2))
    _cluster(rd.Grid(16, 16, inp.default_params()), 1)
    g.set_state(x, -x)
    h.set_state(x, -x)
    before = rd.launch_count()
    g.run(T)
    made = rd.launch_count() - before
    assert made == launches if launches else made > 1
    for t in range(0, T, 101):
        h.run(min(101, T - t), variant="generic")
    assert torch.equal(g.u, h.u) and torch.equal(g.v, h.v)


@pytest.mark.parametrize("shape,every,launches", [((256, 256), 1, 10), ((512, 256), 4, 10), ((64, 64), 30, 10)])
def test_snapshots_between_cluster_and_launches(rd, shape, every, launches):
    """Every few steps kept: a launch each, written where they are kept; many: a cluster launch each."""
    x = torch.from_numpy(inp.uniform_field(48, *shape)).float().cuda()
    g, h = (rd.Grid(*shape, inp.default_params()) for _ in range(2))
    g.set_state(x, -x)
    h.set_state(x, -x)
    before = rd.launch_count()
    us, vs = g.run_snapshots(10 * every, every, out="device")
    assert rd.launch_count() - before == launches
    for s in range(11):
        assert torch.equal(us[s], h.u) and torch.equal(vs[s], h.v), s
        h.run(every, variant="generic")


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
    x, y = (torch.from_numpy(inp.uniform_field(s, *shape)).float().cuda() for s in (44, 45))
    g = rd.Grid(*shape, _gene(reaction), reaction=reaction, boundary=boundary)
    g.set_state(x, y)
    _cluster(g, 9, give_up=1)
    torch.cuda.synchronize()
    assert torch.isnan(g.u).all() and torch.isnan(g.v).all()
    out = []
    for run in (lambda: _cluster(g, 9), lambda: g.run(9, variant="generic")):
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
