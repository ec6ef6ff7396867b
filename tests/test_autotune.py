"""The autotuner's choices, with the measurement and the GPU faked: what it
measures, repeats, counts, returns and caches."""
import types

import pytest

from paper_1807_00672_gb300 import autotune, inputs


@pytest.fixture
def fake(monkeypatch, tmp_path):
    torch = pytest.importorskip("torch")
    monkeypatch.setenv("SWE_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "gpu")
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(multi_processor_count=152))
    seen = []

    def measure(cases, precision, shape, steps=32, warmup=16):
        seen.append((len(cases), shape))
        return 1.0 if shape == autotune.DEFAULT else 2.0 + shape[0]

    monkeypatch.setattr(autotune, "measure", measure)
    return seen


def small_cases(n):
    return [inputs.stoker_case(nx=4 + i, ny=3) for i in range(n)]


def test_the_librarys_own_choice_is_measured_and_returned(fake):
    r = autotune.tune(small_cases(1))
    assert (r["tile"], r["cells_per_thread"], r["stages"], r["halo_schedule"]) == (0, 0, 0, 0)
    assert [s for _, s in fake] == list(autotune.CANDIDATES)
    assert autotune.tune(small_cases(1))["cached"]


def test_a_sample_says_nothing_about_the_librarys_choice(fake):
    cases = small_cases(3)
    cells = sum(c.mesh.n_tris for c in cases)
    for kw in (dict(key_cells=10 * cells, key_scenarios=30), dict(key_cells=cells + 1),
               dict(key_scenarios=4)):
        fake.clear()
        r = autotune.tune(cases, use_cache=False, **kw)
        assert r["tile"] > 0 and autotune.DEFAULT not in [s for _, s in fake]
        assert r["sample_cells"] == cells
    # repeated up to the whole's cells, or to where every ensemble runs in as many waves
    fake.clear()
    autotune.tune(cases, use_cache=False, key_cells=10 * cells)
    assert fake[0][0] == 30


def test_keys_hold_the_callers_scenarios(fake):
    cases = small_cases(3)
    cells = sum(c.mesh.n_tris for c in cases)
    assert "|s3|" in autotune.tune(cases, use_cache=False, key_cells=50 * cells)["key"]
    assert "|s7|" in autotune.tune(cases, use_cache=False, key_cells=50 * cells, key_scenarios=7)["key"]
    # a shape found for a mesh that cannot stay on chip is not taken for one that can
    for prec, n in autotune.ON_CHIP_CELLS.items():
        assert autotune.problem_key("gpu", prec, n, 1) != autotune.problem_key("gpu", prec, n + 1, 1)
