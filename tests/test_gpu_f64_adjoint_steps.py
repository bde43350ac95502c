"""The FP64 adjoint's single-step reverse sweep (no depth asked for) against its pipeline (depth 2) at
the edges of a warp's 64 columns, with one and several rows a warp, widths too narrow for its records
(which take the pipeline), and every model.  The co-states are formed alike, so they agree bit for bit.
The gene's sums are added in another order: on either side a term passes through fewer than 100
additions (a lane's rows, its group or warp, one a launch, 70 records of a thread, 8 levels) and 4
roundings of its own, so the two differ by at most 2 x 104 x 2^-53 = 2.4e-14 of the sum of the terms'
magnitudes, which _magnitudes forms from the states and co-states of every step."""
import numpy as np
import pytest
import torch

import rdcnn_inputs as inp

pytestmark = pytest.mark.gpu

SHAPES = [(1, 64), (2, 2), (3, 22), (5, 24), (33, 62), (17, 66), (64, 128), (7, 130), (1030, 258)]
CENN = {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0}


def _around(x, boundary):
    """Sum of the four neighbours."""
    def shift(d, axis):
        n = x.shape[axis]
        i = torch.arange(n, device=x.device) + d
        return x.index_select(axis, i % n if boundary == "periodic" else i.clamp(0, n - 1))
    return shift(-1, 0) + shift(1, 0) + shift(-1, 1) + shift(1, 1)


def _magnitudes(grid, T, gene, reaction, boundary, u0, v0, gu, gv):
    """Sums over steps and cells of the magnitudes of the terms of each gene entry's derivative."""
    states = [(u0, v0)]
    grid.set_state(u0, v0)
    for _ in range(T - 1):
        grid.run(1)
        states.append(grid.state())
    out = dict.fromkeys(("Du", "Dv", "a", "b", "eps", "c"), 0.0)
    for u, v in reversed(states):
        lu, lv, u_, v_ = gu.abs(), gv.abs(), u.abs(), v.abs()
        if reaction == "cenn":
            y = u_.clamp(max=1.0)
            step = {"Du": lu * _around(y, boundary), "c": lu * y}
        else:
            step = {"Du": u_ * (_around(lu, boundary) + 4 * lu), "Dv": v_ * (_around(lv, boundary) + 4 * lv)}
            if reaction == "fhn":
                e, b, a = abs(gene["eps"]), abs(gene["b"]), abs(gene["a"])
                step.update(a=lv * e, b=lv * e * v_, eps=lv * (u_ + b * v_ + a), c=lu * u_)
        for k, t in step.items():
            out[k] += gene["dt"] * float(t.sum())
        gu, gv, _ = grid.adjoint(1, u, v, gu, gv)
    return out


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("boundary,reaction", [("periodic", "fhn"), ("zeroflux", "fhn"), ("zeroflux", "cenn"),
                                               ("periodic", "none")])
def test_single_steps_match_the_pipeline(rd, shape, boundary, reaction):
    gene = dict(CENN) if reaction == "cenn" else inp.default_params()
    f = lambda seed: torch.from_numpy(np.ascontiguousarray(inp.uniform_field(seed, *shape))).double().cuda()  # noqa: E731
    u0, v0, gu, gv = f(61), 0.7 * f(62), f(63), f(64)
    for T in (1, 2, 11):
        out = []
        for k in (0, 2):
            g = rd.Grid(*shape, gene, dtype=torch.float64, reaction=reaction, boundary=boundary)
            g.set_tune(k=k)
            out.append(g.adjoint(T, u0, v0, gu, gv))
        (du, dv, gp), (eu, ev, ep) = out
        assert torch.equal(du, eu) and torch.equal(dv, ev), T
        size = _magnitudes(g, T, gene, reaction, boundary, u0, v0, gu, gv)
        for name in gp:
            assert abs(gp[name] - ep[name]) <= 2.4e-14 * size[name], (T, name, gp[name], ep[name], size[name])
