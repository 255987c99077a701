"""How many systems an apply call has: the length of its frequency array, whatever that array's shape, and vectors
of any other size are refused (host checks of the binding)."""
import types

import numpy as np
import pytest

from paper_1705_08849_gb300 import fit

torch = pytest.importorskip("torch")
NE = 12


def _vec(nb):
    return types.SimpleNamespace(is_cuda=True, dtype=torch.complex64, is_contiguous=lambda: True, numel=lambda: NE * nb,
                                 data_ptr=lambda: 0)


def _apply(monkeypatch, omega, nb):
    monkeypatch.setattr(fit, "lib", lambda: types.SimpleNamespace(fit_capture_hold=lambda s, t: 0))
    seen = []
    fit._call_apply(lambda *a: seen.append(a) or 0, "fit_apply", None, NE, omega, _vec(nb), _vec(nb), fit.FIT_C64, 5)
    return seen[0][1]


@pytest.mark.parametrize("omega,nb", [(3.0, 1), (np.float64(3), 1), (np.array(3.0), 1), ([3.0, 4.0], 2), ((3.0,), 1),
                                      (np.ones(3), 3), (np.ones((1, 3)), 1), (np.ones((2, 3)), 2), (np.ones((3, 1)), 3),
                                      (np.ones((2, 3), order="F"), 2)])
def test_systems_of_a_call(monkeypatch, omega, nb):
    assert _apply(monkeypatch, omega, nb) == nb
    for other in {1, 2, 3, 6} - {nb}:
        with pytest.raises(ValueError):
            _apply(monkeypatch, omega, other)
