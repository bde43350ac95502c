"""The FP64 adjoint's single-step reverse sweep (no depth asked for) against its pipeline (depth 2) at
the edges of a warp's 64 columns, with one and several rows a warp, widths too narrow for its records
(which take the pipeline), and every model.  The co-states are formed alike, so they agree bit for bit;
the gene's sums are added in another order: 1e-12 of the sum of magnitudes bounds 2^16 FP64 additions
(2^16 x 2^-53 = 7e-12 at worst, its square root in practice)."""
import numpy as np
import pytest
import torch

import rdcnn_inputs as inp

pytestmark = pytest.mark.gpu

SHAPES = [(1, 64), (2, 2), (3, 22), (5, 24), (33, 62), (17, 66), (64, 128), (7, 130), (1030, 258)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("boundary,reaction", [("periodic", "fhn"), ("zeroflux", "fhn"), ("zeroflux", "cenn"),
                                               ("periodic", "none")])
def test_single_steps_match_the_pipeline(rd, shape, boundary, reaction):
    gene = {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0} if reaction == "cenn" \
        else inp.default_params()
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
        scale = max(1.0, T * shape[0] * shape[1] * 0.1)
        for name in gp:
            assert abs(gp[name] - ep[name]) <= 1e-12 * scale, (name, gp[name], ep[name])
