"""The Python binding's own logic, against a stand-in for the library (no GPU)."""
import ctypes

import numpy as np
import pytest

from paper_0903_3852_gb300 import sde


class FakeLib:
    """Counts the rows of runs as the library does and fills mean with 0, 1, ..."""

    def __init__(self):
        self.rows, self.calls, self.every = 0, 0, 0

    def sde_create(self, cfg, h):
        self.every = cfg._obj.sample_every
        h._obj.value = 1
        return sde.SDE_OK

    def sde_destroy(self, h):
        pass

    def sde_run_ensemble(self, h, r, stream):
        n = r._obj.n_end - r._obj.n_begin
        self.rows = -(-n // self.every) + 1 if self.every > 0 else 0
        return sde.SDE_OK

    def sde_observables(self, h, rows, cap, n):
        self.calls += 1
        if cap < 0:
            return sde.SDE_ERR_INVALID_ARG
        for i in range(min(cap, self.rows)):
            rows[i].mean = i
        n._obj.value = self.rows
        return sde.SDE_OK

    def sde_last_error(self):
        return b"rows/capacity"


@pytest.fixture
def fake(monkeypatch):
    f = FakeLib()
    monkeypatch.setattr(sde, "lib", lambda: f)
    monkeypatch.setattr(sde, "_ptr", lambda t: None)
    monkeypatch.setattr(sde, "_stream", lambda s: None)
    return f


def kuramoto_config(every):
    cfg = sde.Config()
    cfg.model, cfg.n_osc, cfg.n_replicas, cfg.sample_every = sde.SDE_KURAMOTO_MEANFIELD, 8, 1, every
    return cfg


def test_an_ensemble_made_from_a_config_runs_and_reports(fake):
    ens = sde.Ensemble(kuramoto_config(10))
    ens.run_kuramoto(5, 30, None, None, None)
    assert ens.observables()["mean"].tolist() == [0, 1, 2, 3] and fake.calls == 1
    assert ens.observables(capacity=2)["mean"].tolist() == [0, 1]
    assert len(ens.observables(capacity=9)) == 4


def test_rows_of_a_run_made_through_the_c_functions(fake):
    ens = sde.Ensemble(kuramoto_config(10))
    r = sde.RunDesc()
    r.n_begin, r.n_end = 0, 100
    assert sde.lib().sde_run_ensemble(ens._h, ctypes.byref(r), None) == sde.SDE_OK
    assert ens.observables()["mean"].tolist() == list(range(11))
    ens.run_kuramoto(0, 10, None, None, None)
    assert len(ens.observables()) == 2
    assert isinstance(ens.observables(), np.ndarray)


def test_a_negative_capacity_is_refused_by_the_library(fake):
    ens = sde.Ensemble(kuramoto_config(10))
    with pytest.raises(sde.SDEError):
        ens.observables(capacity=-1)
