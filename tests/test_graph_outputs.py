"""The binding's output tensors of evaluate_graph belong to the particles they were made for.

Runs on the CPU: the library's call is a stand-in that notes the pointers it is given.
"""
import pytest

from paper_2005_12351_gb300 import fmm


class Call:
    def __init__(self):
        self.outputs = []

    def __call__(self, handle, p, theta, want_phi, want_field, phi, field):
        self.outputs.append((phi.value if phi else None, field.value if field else None))
        return 0


@pytest.mark.parametrize("want", [(True, True), (True, False), (False, True)])
def test_another_number_of_particles_takes_other_outputs(monkeypatch, want):
    call = Call()
    monkeypatch.setattr(fmm, "lib", lambda: type("Lib", (), {"fmm_evaluate_graph": call})())
    t = fmm.FMMTree.__new__(fmm.FMMTree)
    t._h, t.device = None, "cpu"
    kept = []
    for n in (1000, 60, 1000, 5000, 5000):
        t.n = n
        out = t.evaluate_graph(4, 0.5, *want)
        for v, shape, w in zip(out, ((n,), (n, 3)), want):
            assert (v is not None) == w
            assert v is None or tuple(v.shape) == shape
        assert call.outputs[-1] == tuple(None if v is None else v.data_ptr() for v in out)
        kept.append(out)
    assert call.outputs[-1] == call.outputs[-2]         # the same particles: the same tensors, one graph
