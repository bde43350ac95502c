"""The launch-shape tuner's choice among its candidates (host logic, a grid that only records calls):
the library's own choice is one of them, timed with nothing tuned, and stays in force when it wins."""
import pytest

torch = pytest.importorskip("torch")


class _Grid:
    reaction, boundary = "fhn", "periodic"

    def __init__(self, nn, nm, dtype):
        self.nn, self.nm, self.dtype = nn, nm, dtype
        self.tune = (9, 9)
        self.last = None

    def set_tune(self, k=0, rows=0):
        self.tune = (k, rows)

    def run(self, T, variant="auto", k=0):
        self.last = (variant, k, *self.tune)


def _tuned(monkeypatch, grid, cost):
    from paper_2102_10340_gb300 import autotune

    def fake(fn, reps=2):
        fn()
        return cost(*grid.last)

    monkeypatch.setattr(autotune, "_time", fake)
    monkeypatch.setattr(autotune, "_cache", {})
    return autotune.tune_grid(grid)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64, torch.bfloat16])
def test_the_library_s_own_choice_can_win(monkeypatch, dtype):
    g = _Grid(64, 64, dtype)
    best = _tuned(monkeypatch, g, lambda variant, k, tk, tr: 1.0 if (variant, k, tk, tr) == ("auto", 0, 0, 0) else 2.0)
    assert (best["variant"], best["k"], best["rows"]) == ("auto", 0, 0)
    assert g.tune == (0, 0)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("rows", [1, 2])
def test_short_single_step_strips_are_tried(monkeypatch, dtype, rows):
    g = _Grid(512, 512, dtype)
    best = _tuned(monkeypatch, g, lambda variant, k, tk, tr: 1.0 if (variant, tr) == ("step1", rows) else 2.0)
    assert (best["variant"], best["k"], best["rows"]) == ("step1", 1, rows)
    assert g.tune == (1, rows)


def test_a_faster_shape_still_wins(monkeypatch):
    g = _Grid(512, 512, torch.float32)
    best = _tuned(monkeypatch, g, lambda variant, k, tk, tr: 1.0 if (variant, k, tr) == ("temporal", 6, 64) else 2.0)
    assert (best["variant"], best["k"], best["rows"]) == ("temporal", 6, 64) and g.tune == (6, 64)
