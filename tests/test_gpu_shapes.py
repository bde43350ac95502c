"""Launch shapes and stretches that AUTO chooses: runs end in (u, v) whatever the number of launches,
device snapshots written by the steps themselves, statistics with and without whole vectors, and FP32
batches of mixed sizes, each against the plain path."""
import numpy as np
import pytest
import torch

import rdcnn_inputs as inp
from _util import gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 260), (45, 300), (301, 299), (700, 264), (1030, 520)])
@pytest.mark.parametrize("boundary", ["periodic", "zeroflux"])
def test_any_number_of_steps(rd, shape, boundary):
    x, y = inp.uniform_field(71, *shape), 0.7 * inp.uniform_field(72, *shape)
    for T in (1, 2, 3, 5, 8, 9, 17, 41):
        a, b = (gpu_run(rd, x, y, inp.default_params(), T, torch.float32, v, boundary=boundary) for v in ("auto", "generic"))
        assert (a[0] == b[0]).all() and (a[1] == b[1]).all(), T


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64, torch.bfloat16])
@pytest.mark.parametrize("shape", [(96, 300), (64, 64), (37, 261)])
@pytest.mark.parametrize("T,every", [(20, 20), (23, 7), (12, 1), (5, 9), (30, 4)])
@pytest.mark.parametrize("offset", [0, 1])
def test_device_snapshots(rd, dtype, shape, T, every, offset):
    """Against copies of the state taken between runs of `every` steps (16-bit: the same launches).
    offset: the arrays one element off an aligned address."""
    n = T // every + 1
    g = rd.Grid(*shape, inp.default_params(), dtype=dtype)
    x = torch.from_numpy(inp.uniform_field(73, *shape)).to(dtype).cuda()
    g.init(x)
    cells = n * shape[0] * shape[1]
    base = [torch.full((cells + 2,), 7.0, dtype=dtype, device="cuda") for _ in range(2)]
    us, vs = (t[offset:offset + cells].view(n, *shape) for t in base)
    g.run_snapshots(T, every, out="device", buffers=(us, vs))
    h = rd.Grid(*shape, inp.default_params(), dtype=dtype)
    h.init(x)
    for s in range(n):
        assert torch.equal(us[s], h.u) and torch.equal(vs[s], h.v), s
        h.run(every if s + 1 < n else T % every)
    assert torch.equal(g.u, h.u) and torch.equal(g.v, h.v)
    assert all(float(t[-1]) == 7.0 and (offset == 0 or float(t[0]) == 7.0) for t in base)


@pytest.mark.parametrize("shape", [(1, 4), (9, 124), (16, 128), (1000, 132), (5, 131), (70, 516)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64, torch.float16])
@pytest.mark.parametrize("offset", [0, 1])
def test_statistics_with_and_without_vectors(rd, shape, dtype, offset):
    """FP32: a lane adds up to 20 values (516 columns), then 5 levels of a tree, 25 roundings of 6e-8 of sums of
    positive terms or of values in [-1, 1]: 1e-5 relative or absolute holds both; FP64 1e-12."""
    cells = shape[0] * shape[1]
    base = [torch.zeros(cells + 1, dtype=dtype, device="cuda") for _ in range(2)]
    u, v = (t[offset:offset + cells].view(shape) for t in base)
    u.copy_(torch.from_numpy(inp.uniform_field(74, *shape)))
    v.copy_(torch.from_numpy(inp.uniform_field(75, *shape)))
    got = rd.rdcnn.grid_summary(u, v, 0.8).numpy() if hasattr(rd, "rdcnn") else rd.grid_summary(u, v, 0.8).numpy()
    a, b = u.double().cpu().numpy(), v.double().cpu().numpy()
    grad = np.abs(np.roll(a, -1, 0) - a) + np.abs(np.roll(a, -1, 1) - a)
    want = [a.mean(), a.var(), a.min(), a.max(), b.mean(), b.var(), grad.mean(), (grad > 0.8).mean()]
    tol = 1e-12 if dtype == torch.float64 else 1e-5
    np.testing.assert_allclose(got[:7], want[:7], rtol=tol, atol=tol)
    assert abs(got[7] - want[7]) <= 2.0 / cells  # a gradient within rounding of the threshold


@pytest.mark.parametrize("sides", [(32,), (32, 300), (128, 256, 512), (64, 1024, 96)])
@pytest.mark.parametrize("T", [1, 3, 16, 29])
def test_batches_of_mixed_sizes(rd, sides, T):
    specs = [{"nn": s, "nm": s + 4 * i, "params": inp.default_params(Du=0.03 * (i + 1))} for i, s in enumerate(sides * 2)]
    b = rd.Batch(specs, dtype=torch.float32)
    xs = [torch.from_numpy(inp.uniform_field(76 + i, s["nn"], s["nm"])).float().cuda() for i, s in enumerate(specs)]
    for i, x in enumerate(xs):
        b.set_state(i, x, -x)
    b.run(T)
    for i, (s, x) in enumerate(zip(specs, xs)):
        ref = gpu_run(rd, x.double().cpu().numpy(), -x.double().cpu().numpy(), s["params"], T, torch.float32, "generic")
        assert all((t.cpu().numpy() == r).all() for t, r in zip(b.state(i), ref)), i


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64, torch.bfloat16])
def test_batch_state_copies(rd, dtype):
    """States from tensors of every kind a caller may hold: the same plane twice, whole and offset
    views, another type, transposed, on the host, and the instance's own planes (u is set first)."""
    nn, nm = 33, 52
    specs = [{"nn": nn, "nm": nm, "params": inp.default_params()}]
    x, y = (torch.from_numpy(inp.uniform_field(s, nn, nm)).to(dtype).cuda() for s in (81, 82))
    off = torch.zeros(nn * nm + 1, dtype=dtype, device="cuda")[1:].view(nn, nm)
    off.copy_(y)
    for a, b in ((x, x), (x, y), (x, off), (off, x), (x.double(), y.float()), (x, y.t().contiguous().t()), (x.cpu(), y.cpu())):
        t = rd.Batch(specs, dtype=dtype)
        t.set_state(0, a, b)
        assert torch.equal(t.state(0)[0], a.to("cuda", dtype)) and torch.equal(t.state(0)[1], b.to("cuda", dtype))
    t.set_state(0, x, y)
    t.set_state(0, t.state(0)[1], t.state(0)[0])
    assert torch.equal(t.state(0)[0], y) and torch.equal(t.state(0)[1], y)
    with pytest.raises(RuntimeError):
        t.set_state(0, x[:, :-4].contiguous(), y[:, :-4].contiguous())


def test_training_results_outlive_later_calls(rd):
    """The final state returned by RDCNNFunction keeps its values, and the graph its gradients, when
    the outputs are written over and other calls run in between."""
    f = lambda seed: torch.from_numpy(inp.uniform_field(seed, 40, 64)).float().cuda()  # noqa: E731
    th = torch.tensor([inp.default_params()[k] for k in rd.GRAD_NAMES], dtype=torch.float64)
    out = []
    for disturb in (False, True):
        u0, v0, t = f(91).requires_grad_(True), f(92).requires_grad_(True), th.clone().requires_grad_(True)
        u, v = rd.RDCNNFunction.apply(u0, v0, t, 30)
        loss = (u * f(93)).sum() + (v * f(94)).sum()
        kept = u.detach().clone()
        if disturb:
            with torch.no_grad():
                rd.RDCNNFunction.apply(f(95), f(96), th, 7)
                u.detach().zero_()
        out.append((kept, *torch.autograd.grad(loss, (u0, v0, t))))
    assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65])
def test_number_of_instances(rd, n):
    """Both sides of the number of instances whose table travels with the launch."""
    specs = [{"nn": 5 + i % 7, "nm": 4 * (1 + i % 40), "params": inp.default_params(Du=0.002 * (i + 1))} for i in range(n)]
    b = rd.Batch(specs, dtype=torch.float32, boundary="zeroflux")
    xs = [torch.from_numpy(inp.uniform_field(100 + i, s["nn"], s["nm"])).float().cuda() for i, s in enumerate(specs)]
    for i, x in enumerate(xs):
        b.set_state(i, x, -x)
    b.run(11)
    for i, (s, x) in enumerate(zip(specs, xs)):
        ref = gpu_run(rd, x.double().cpu().numpy(), -x.double().cpu().numpy(), s["params"], 11, torch.float32, "generic",
                      boundary="zeroflux")
        assert all((t.cpu().numpy() == r).all() for t, r in zip(b.state(i), ref)), i


def test_captured_states_and_odd_runs(rd):
    """Setting a state and a run that ends in the scratch planes, recorded into the caller's graph."""
    nn, nm = 40, 300
    x, y = (torch.from_numpy(inp.uniform_field(s, nn, nm)).float().cuda() for s in (83, 84))
    g, h = (rd.Grid(nn, nm, inp.default_params()) for _ in range(2))
    for t in (g, h):
        t.set_state(x, y).run(3, variant="step1")
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        g.set_state(y, x).run(5, variant="step1")
    h.set_state(y, x).run(5, variant="step1")
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(g.u, h.u) and torch.equal(g.v, h.v)


@pytest.mark.parametrize("boundary,reaction", [("periodic", "fhn"), ("zeroflux", "fhn"), ("periodic", "cenn")])
def test_strips_beyond_l2(rd, boundary, reaction):
    """Strips of depths 1 to 4 from six million cells on: their lengths, whole waves at depths 3 and 4, and
    the bits of the one-thread-per-cell kernel."""
    gene = {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0} if reaction == "cenn" \
        else inp.default_params()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nn, nm = 2600, 2400  # 20 bands
    x = torch.rand((nn, nm), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda") * 2 - 1
    ref = rd.Grid(nn, nm, gene, boundary=boundary, reaction=reaction)
    ref.set_state(x, -x).run(12, variant="generic")
    for k in (1, 2, 3, 4):
        g = rd.Grid(nn, nm, gene, boundary=boundary, reaction=reaction)
        rows = g.plan("temporal", k)["rows"]
        if k < 3:
            assert rows == (10, 12)[k - 1]
        else:
            assert any(rows == -(-nn // (p * sms // 20)) for p in ((12,) if k == 3 else (4, 8, 12, 16, 20)))
        g.set_state(x, -x).run(12, variant="temporal", k=k)
        assert torch.equal(g.u, ref.u) and torch.equal(g.v, ref.v), k
    small = rd.Grid(2400, 2400, gene, boundary=boundary, reaction=reaction)  # 5.76 million: the launch model
    assert small.plan("temporal", 1)["rows"] != 10


@pytest.mark.parametrize("shape,T,launches", [((512, 512), 9, 2), ((1024, 1024), 10, 2), ((5000, 5000), 4, 1),
                                              ((2600, 2400), 8, 2), ((509, 515), 9, 2)])
def test_launches_of_short_stretches(rd, shape, T, launches):
    """Few deep launches, or one and a copy of the state, where more launches would cost more; the same bits."""
    x = torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda") * 2 - 1
    g, h = (rd.Grid(*shape, inp.default_params()) for _ in range(2))
    g.set_state(x, -x)
    before = rd.launch_count()
    g.run(T)
    assert rd.launch_count() - before == launches
    h.set_state(x, -x).run(T, variant="generic")
    assert torch.equal(g.u, h.u) and torch.equal(g.v, h.v)


@pytest.mark.parametrize("shape,rows,want", [((256, 256), 0, ("step1", 1)), ((256, 256), 15, ("step1", 1)),
                                             ((256, 256), 16, ("temporal", 4)), ((1024, 1024), 16, ("step1", 1)),
                                             ((1024, 1024), 128, ("temporal", 4)), ((300, 301), 64, ("generic", 1))])
def test_fp64_strips_asked_for(rd, shape, rows, want):
    """AUTO with a strip length but no depth: single steps, or the pipeline where the strips are few and long."""
    x = torch.from_numpy(inp.uniform_field(87, *shape)).double().cuda()
    g, h = (rd.Grid(*shape, inp.default_params(), dtype=torch.float64) for _ in range(2))
    g.set_tune(k=0, rows=rows)
    plan = g.plan()
    assert (plan["variant"], plan["k"]) == want and (want[0] == "generic" or rows == 0 or plan["rows"] == rows)
    g.set_state(x, -x).run(9)
    h.set_state(x, -x).run(9, variant="generic")
    assert torch.equal(g.u, h.u) and torch.equal(g.v, h.v)
