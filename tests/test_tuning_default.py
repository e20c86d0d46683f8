"""Host logic of the autotuner (no GPU): the library default is among the
timed configurations, and a choice is kept for the relaxation times it was
timed with."""
import pytest

from paper_1405_6162_gb300 import tuning
from paper_1405_6162_gb300 import lattice as lattice_module

DIMS = (64, 64, 80)


class _Lattice:
    """Stands in for the lattice; ``seconds`` of a configuration are a step's."""
    seconds = staticmethod(lambda config, params: 1.0)

    def __init__(self, params):
        self.params = params

    @classmethod
    def from_params(cls, dims, params, precision):
        return cls(params)

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        pass

    def init(self, phi0):
        pass


@pytest.fixture(autouse=True)
def _fakes(tmp_path, monkeypatch):
    monkeypatch.setattr(tuning, "CACHE", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(tuning, "_gpu_name", lambda: "probe-gpu")
    monkeypatch.setattr(lattice_module, "Lattice", _Lattice)
    monkeypatch.setattr(tuning, "time_config", lambda lat, cfg, steps=5: _Lattice.seconds(tuple(cfg), lat.params))


def _fastest(monkeypatch, by_tau_g):
    monkeypatch.setattr(_Lattice, "seconds",
                        staticmethod(lambda cfg, p: 1.0 if cfg == by_tau_g[p["tau_g"] == 1.0] else 2.0))


@pytest.mark.parametrize("precision", ["fp32_shifted", "fp64", "fp64_df"])
def test_the_untouched_library_is_never_slower_than_the_choice(monkeypatch, precision):
    _fastest(monkeypatch, {True: tuning.DEFAULT, False: tuning.DEFAULT})
    best, table = tuning.autotune(DIMS, precision, {"tau": 1.0, "tau_g": 1.0}, None)
    assert best == tuning.DEFAULT
    assert {c[0] for c, _ in table} >= {"auto", "two_pass"}
    # the reduced form keeps another state: the general default is not offered for it
    _, table = tuning.autotune(DIMS, precision, {"tau": 1.0, "tau_g": 1.0}, None, families=("taug1",))
    assert {c[0] for c, _ in table} == {"taug1"}


def test_a_choice_is_not_used_for_other_relaxation_times(monkeypatch):
    one, other = {"tau": 0.8, "tau_g": 1.0}, {"tau": 0.8, "tau_g": 0.9}
    bulk = ("bulk", 3, 2, 16)
    _fastest(monkeypatch, {True: tuning.DEFAULT, False: bulk})
    assert tuning.ensure_tuned(DIMS, "fp32_shifted", one, None) == tuning.DEFAULT
    assert tuning.ensure_tuned(DIMS, "fp32_shifted", other, None) == bulk
    assert tuning.ensure_tuned(DIMS, "fp32_shifted", one, None) == tuning.DEFAULT
    assert tuning.bench_config(DIMS, "fp32_shifted", params=other) == bulk
    assert tuning.bench_config(DIMS, "fp32_shifted", params={"tau": 1.0, "tau_g": 0.9}) == tuning.DEFAULT
    # without parameters: the last one tuned
    assert tuning.bench_config(DIMS, "fp32_shifted") == bulk
    assert tuning.cached_table(DIMS, "fp32_shifted")["config"] == list(bulk)


def test_the_default_steps_summary_is_current():
    import bench
    assert bench._profile_value("step_default_fp32_256cubed", "dram_bytes_per_step") is not None
