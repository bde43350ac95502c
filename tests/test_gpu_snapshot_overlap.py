"""Device snapshots whose arrays share memory with the state or with one another: the bound planes are
slots of the arrays (the state then ends where its last snapshot lies), or one array takes both fields.
The state runs on as if each snapshot were copied out after its step."""
import ctypes

import pytest
import torch

import rdcnn_inputs as inp

pytestmark = pytest.mark.gpu

SHAPES = [(64, 64), (300, 300), (96, 400), (37, 401)]


def _reference(rd, shape, dtype, x, y, n, every):
    g = rd.Grid(*shape, inp.default_params(), dtype=dtype)
    g.set_state(x, y)
    out = [(x, y)]
    for _ in range(n - 1):
        g.run(every)
        out.append(g.state())
    return out


def _start(shape, dtype):
    return [torch.from_numpy(inp.uniform_field(s, *shape)).to(dtype).cuda() for s in (85, 86)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("every", [1, 3, 8])
@pytest.mark.parametrize("slot", [0, 2, 4])
def test_state_planes_are_a_slot(rd, shape, dtype, every, slot):
    """A slot that is the state is overwritten by later steps: the others hold their snapshots."""
    from paper_2102_10340_gb300 import _lib as L

    n, (nn, nm) = 5, shape
    x, y = _start(shape, dtype)
    us, vs = (torch.zeros((n, nn, nm), dtype=dtype, device="cuda") for _ in range(2))
    us[slot], vs[slot] = x, y
    g = rd.Grid(nn, nm, inp.default_params(), dtype=dtype)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    vp = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    L.check(g.lib.rdcnn_bind(g.h, vp(us[slot]), vp(vs[slot]), vp(g.workspace),
                             g.workspace.numel() * g.workspace.element_size(), stream))
    L.check(g.lib.rdcnn_run_snapshots(g.h, (n - 1) * every, every, vp(us), vp(vs), 1, None, 0))
    ref = _reference(rd, shape, dtype, x, y, n, every)
    for s in range(n):
        a, b = ref[n - 1] if s == slot else ref[s]
        assert torch.equal(us[s], a) and torch.equal(vs[s], b), s


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("every", [1, 8])
@pytest.mark.parametrize("shift", [0, 1])
def test_arrays_that_overlap(rd, shape, dtype, every, shift):
    """One array for both fields (v is copied last), and v's slot s in the place of u's slot s + 1
    (which the next snapshot then takes)."""
    n, (nn, nm) = 4, shape
    x, y = _start(shape, dtype)
    g = rd.Grid(nn, nm, inp.default_params(), dtype=dtype)
    g.set_state(x, y)
    base = torch.zeros((n + shift, nn, nm), dtype=dtype, device="cuda")
    g.run_snapshots((n - 1) * every, every, out="device", buffers=(base[:n], base[shift:]))
    ref = _reference(rd, shape, dtype, x, y, n, every)
    assert torch.equal(g.u, ref[-1][0]) and torch.equal(g.v, ref[-1][1])
    for s in range(n + shift):
        want = ref[s][0] if shift and s < n else ref[s - shift][1]
        assert torch.equal(base[s], want), s
