"""The frequency array that a captured call reads at every replay lives as long as the graph, whatever the
caller passed: host logic of the binding, with a stand-in for the runtime's part (which stream is being captured,
which graphs are gone)."""
import gc
import types
import weakref

import numpy as np
import pytest

from paper_1705_08849_gb300 import build, fit


@pytest.fixture
def runtime(monkeypatch):
    """A library whose streams 7 and 8 are being captured, and weak references to every array made for a call."""
    build.build()
    rt = types.SimpleNamespace(graphs={7: [], 8: []}, gone=[], made=[])

    def hold(stream, token):
        stream = getattr(stream, "value", stream)
        rt.graphs.get(stream, []).append(token)
        return int(stream in rt.graphs)

    def released(out, cap):
        n = min(cap, len(rt.gone))
        out[:n] = rt.gone[:n]
        del rt.gone[:n]
        return n

    real = fit.np.ascontiguousarray

    def making(*a, **k):
        out = real(*a, **k)
        rt.made.append(weakref.ref(out))
        return out

    fake = types.SimpleNamespace(fit_capture_hold=hold, fit_capture_released=released, fit_jacobi=lambda *a: 0,
                                 fit_grid_info=lambda g, out: out.__setitem__(3, 12) or 0, fit_last_error=lambda: b"")
    monkeypatch.setattr(fit, "lib", lambda: fake)
    monkeypatch.setattr(fit.np, "ascontiguousarray", making)
    yield rt
    rt.gone += [t for g in rt.graphs.values() for t in g]
    if hasattr(fit, "_hold_for_graph"):
        fit._hold_for_graph(np.zeros(1), 8)  # (takes the released ones out)


def _vec(nb):
    torch = pytest.importorskip("torch")
    return types.SimpleNamespace(is_cuda=True, dtype=torch.complex64, is_contiguous=lambda: True, numel=lambda: 12 * nb,
                                 data_ptr=lambda: 0)


def _apply(omega, nb, stream):
    seen = []
    fit._call_apply(lambda *a: seen.append(a) or 0, "fit_apply", None, 12, omega, _vec(nb), _vec(nb), fit.FIT_C64, stream)
    return seen[0]


@pytest.mark.parametrize("omega", [3.0, [3.0, 4.0], np.array([3, 4]), np.array([3.0, 9.0, 4.0])[::2]])
def test_a_temporary_lives_until_its_graphs_are_gone(runtime, omega):
    nb = np.size(omega)
    args = _apply(omega, nb, 7)
    assert args[1] == nb
    gc.collect()
    alive = [r() for r in runtime.made if r() is not None]
    assert any(a.__array_interface__["data"][0] == args[2] for a in alive)
    del alive
    runtime.gone += runtime.graphs[7]
    _apply([1.0], 1, 8)
    gc.collect()
    assert not any(r() is not None and r().__array_interface__["data"][0] == args[2] for r in runtime.made[:-1])


def test_the_callers_own_array_is_held_and_read_in_place(runtime):
    own = np.array([3.0, 4.0])
    ref, at = weakref.ref(own), own.__array_interface__["data"][0]
    assert _apply(own, 2, 7)[2] == at
    del own
    gc.collect()
    assert ref() is not None
    runtime.gone += runtime.graphs[7]
    _apply([1.0], 1, 8)
    gc.collect()
    assert ref() is None


def test_nothing_is_kept_outside_a_capture(runtime):
    own = np.array([3.0])
    ref = weakref.ref(own)
    _apply(own, 1, 5)
    del own
    gc.collect()
    assert ref() is None


def test_jacobi_holds_its_frequencies_too(runtime):
    fit.fit_jacobi(None, [3.0], _vec(1), _vec(1), fit.FIT_C64, 7)
    gc.collect()
    assert any(r() is not None for r in runtime.made)
