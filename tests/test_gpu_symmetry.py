"""FP64 grids on the torus: the neighbour sum (n + s) + (w + e) is unchanged by a reflection of the rows or
of the columns, so a mirror-symmetric start stays mirror-symmetric bit for bit in every variant, in
batches and in the adjoint's co-states.  (FP32 and 16-bit tori group the sum otherwise and keep the
symmetry up to rounding only.)"""
import pytest
import torch

import rdcnn_inputs as inp

pytestmark = pytest.mark.gpu

CENN = {"dt": 0.1, "a": 0.0, "b": 0.0, "eps": 0.0, "c": 1.3, "Du": 0.2, "Dv": 0.0}
REACTIONS = ["fhn", "none", "cenn"]


def _even(seed, nn, nm):
    """A plane that both reflections leave as it is."""
    x = torch.from_numpy(inp.uniform_field(seed, nn, nm)).double().cuda()
    i, j = torch.arange(nn, device="cuda"), torch.arange(nm, device="cuda")
    return x[torch.minimum(i, nn - 1 - i)][:, torch.minimum(j, nm - 1 - j)].contiguous()


def _gene(reaction):
    return CENN if reaction == "cenn" else inp.default_params()


def _assert_even(*planes):
    for t in planes:
        assert torch.isfinite(t).all()
        assert torch.equal(t, t.flip(0)) and torch.equal(t, t.flip(1))


ANY_ROWS = [("auto", 0), ("auto", 3), ("generic", 0)]
VECTOR_ROWS = [("step1", 0)] + [("temporal", k) for k in (1, 2, 3, 4)] + [("temporal2", k) for k in (2, 3, 4)]


@pytest.mark.parametrize("reaction", REACTIONS)
@pytest.mark.parametrize("shape,variant,k", [(s, *v) for s in ((64, 128), (7, 250)) for v in ANY_ROWS + VECTOR_ROWS]
                         + [((45, 67), *v) for v in ANY_ROWS])
def test_runs_keep_a_mirrored_state(rd, reaction, shape, variant, k):
    g = rd.Grid(*shape, _gene(reaction), dtype=torch.float64, reaction=reaction)
    g.set_state(_even(1, *shape), 0.7 * _even(2, *shape)).run(37, variant=variant, k=k)
    _assert_even(g.u, g.v)


@pytest.mark.parametrize("reaction", REACTIONS)
@pytest.mark.parametrize("k", [0, 1, 2, 3, 4])
def test_batches_keep_a_mirrored_state(rd, reaction, k):
    specs = [{"nn": 20 + i, "nm": 64 + 30 * i, "params": _gene(reaction)} for i in range(3)]
    b = rd.Batch(specs, dtype=torch.float64, reaction=reaction)
    b.set_tune(k=k)
    for i, s in enumerate(specs):
        b.set_state(i, _even(3 + i, s["nn"], s["nm"]), 0.7 * _even(6 + i, s["nn"], s["nm"]))
    b.run(21)
    for i in range(3):
        _assert_even(*b.state(i))


@pytest.mark.parametrize("reaction", REACTIONS)
@pytest.mark.parametrize("k,n_checkpoints", [(0, 0), (2, 0), (3, 0), (0, 11)])
def test_adjoints_keep_a_mirrored_costate(rd, reaction, k, n_checkpoints):
    nn, nm = 33, 130
    g = rd.Grid(nn, nm, _gene(reaction), dtype=torch.float64, reaction=reaction)
    g.set_tune(k=k)
    du, dv, _ = g.adjoint(11, _even(9, nn, nm), 0.7 * _even(10, nn, nm), _even(11, nn, nm), _even(12, nn, nm), n_checkpoints)
    _assert_even(du, dv)
