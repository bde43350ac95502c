"""AUTO on planes whose rows are not lane vectors (NM no multiple of the lane width, or planes off
their 16-byte alignment) against the one-thread-per-cell kernel: the same bits, at the edges of a
band (128 columns minus the halos), with wrapped halos wider than the grid, and for every model."""
import pytest
import torch

import rdcnn_inputs as inp
from _util import gpu_run

pytestmark = pytest.mark.gpu

# columns around one band's stored width (112 at depth 8, 120 at depth 4), a band's full width, and tori narrower than a halo
SHAPES = [(1, 1), (3, 5), (1, 7), (2, 1), (5, 113), (19, 119), (37, 121), (64, 127), (9, 129), (70, 243), (530, 261)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("boundary,reaction", [("periodic", "fhn"), ("zeroflux", "fhn"), ("zeroflux", "cenn"),
                                               ("periodic", "none")])
def test_auto_matches_generic_bitwise(rd, shape, dtype, boundary, reaction):
    gene = {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0} if reaction == "cenn" \
        else inp.default_params()
    x, y = inp.uniform_field(31, *shape), 0.7 * inp.uniform_field(32, *shape)
    for T in (1, 7, 22):
        a = gpu_run(rd, x, y, gene, T, dtype, "auto", reaction=reaction, boundary=boundary)
        b = gpu_run(rd, x, y, gene, T, dtype, "generic", reaction=reaction, boundary=boundary)
        assert (a[0] == b[0]).all() and (a[1] == b[1]).all(), T


@pytest.mark.parametrize("dtype,k", [(torch.float32, d) for d in range(1, 9)] + [(torch.float64, 3)])
def test_every_depth_on_misaligned_planes(rd, dtype, k):
    """Planes one element past an aligned address, NM a multiple of the lane width (FP64 planes
    take the one-thread-per-cell kernel whatever the depth)."""
    nn, nm = 45, 132
    x = torch.from_numpy(inp.uniform_field(33, nn, nm)).to(dtype).cuda()
    out = []
    for variant in ("auto", "generic"):
        base = [torch.zeros(1 + nn * nm + 1, dtype=dtype, device="cuda") for _ in range(2)]
        u, v = (t[1:1 + nn * nm].view(nn, nm) for t in base)
        u.copy_(x)
        v.copy_(-x)
        rd.run(u, v, inp.default_params(), 2 * k + 1, variant=variant, k=k)
        assert all(float(t[0]) == 0.0 and float(t[-1]) == 0.0 for t in base)
        out.append((u.clone(), v.clone()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("shape,T,single", [((900, 1), 3, False), ((901, 1), 3, True), ((12600, 14), 24, False),
                                            ((12601, 14), 24, True), ((20000, 15), 24, False), ((23000, 25), 3, True),
                                            ((24000, 26), 3, False), ((2000, 49), 2, None), ((2000, 50), 2, None),
                                            ((2000, 74), 1, None), ((2000, 75), 1, None), ((1100, 189), 2, None),
                                            ((1100, 191), 2, None)])
def test_narrow_grids_take_one_thread_a_cell(rd, shape, T, single):
    """On both sides of the rule: as many launches as steps, or fewer (one or two steps take as many
    launches either way), and the same bits."""
    x, y = (torch.from_numpy(inp.uniform_field(s, *shape)).float().cuda() for s in (34, 35))
    out = []
    for variant in ("auto", "generic"):
        g = rd.Grid(*shape, inp.default_params())
        g.set_state(x, y)
        before = rd.launch_count()
        g.run(T, variant=variant)
        out.append((rd.launch_count() - before, *g.state()))
    assert torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][2], out[1][2])
    assert out[1][0] == T and (single is None or (out[0][0] == T) == single)
