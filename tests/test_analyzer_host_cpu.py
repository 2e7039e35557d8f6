"""What Analyzer takes and keeps, without a device: the launches are replaced by a stand-in that counts candidates."""
import pytest

from paper_2511_15369_b200 import api, assign


class _Launches:
    """analyze_gelu() as the native binding has it: the candidates among `applicable` are run."""

    def __init__(self, applicable=range(100)):
        self.applicable, self.seen = applicable, []

    def analyze_gelu(self, x, in_scale, in_bits, out_scale, out_zp, out_bits, variants, sums, work):
        self.seen.append((list(variants), sums))
        return [(v, 1.0) for v in variants if v in self.applicable]


def _analyzer(monkeypatch, launches, **kw):
    monkeypatch.setattr(api, "native", lambda: launches)
    an = assign.Analyzer(device="cpu", **kw)
    return an, lambda v: an.gelu_layer("x", None, 1e-3, 16, 0.03, 0, variants=v)


@pytest.mark.parametrize("variants", [(2, 0), [2, 0], {0: 1, 2: 1}, iter((2, 0)), (v for v in (2, 0)), range(0, 3, 2)])
def test_candidates_from_any_iterable(monkeypatch, variants):
    an, layer = _analyzer(monkeypatch, _Launches())
    assert sorted(c.variant for c in layer(variants).candidates) == [0, 2]


def test_results_take_attributes(monkeypatch):
    an, layer = _analyzer(monkeypatch, _Launches())
    l = layer((0,))
    l.note = "kept"
    l.candidates[0].note = "kept"


def test_the_capacity_counts_evaluations_alone(monkeypatch):
    """Candidates without integer constants take no room, and a layer that does not fit leaves the layers before it as they are."""
    ls = _Launches(applicable=(0, 1))
    an, layer = _analyzer(monkeypatch, ls, max_evaluations=4)
    assert [c.slot for c in layer((0, 1)).candidates] == [0, 1]
    assert [c.slot for c in layer((0, 5, 1)).candidates] == [2, 3]
    assert layer((5, 6)).candidates == []                      # full, and nothing to evaluate
    for _ in range(3):
        with pytest.raises(RuntimeError):
            layer((0, 1))
    assert len(an.layers) == 3 and an.n_eval == 4
    room = an.sums.data_ptr() + 16 * an.sums.shape[0]
    assert all(at + 16 * len(v) <= room for v, at in ls.seen)  # no launch can write past the buffer
