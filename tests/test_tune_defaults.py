"""The autotuner may keep the constructor's own launch: it is among the candidates of every
precision and path, so a tuned launch is never slower than no tuning, and entries that
older candidates left in the cache are timed again."""
import json

import pytest

from paper_1603_09577_gb300 import tune

DEFAULT = dict(kernel_variant=0, block_rows=0, steps_per_pass=1)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16s"])
@pytest.mark.parametrize("nx", [128, 301])
def test_the_default_launch_is_a_candidate(prec, nx):
    assert DEFAULT in tune.candidates(nx, prec)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("per_cell_K", [False, True])
def test_the_default_launch_is_a_general_candidate(prec, per_cell_K):
    assert DEFAULT in tune.general_candidates(prec, per_cell_K)


@pytest.mark.parametrize("kw", [dict(prec="f64"), dict(prec="f32"), dict(prec="f64", scheme="A")])
def test_the_default_wins_where_it_is_the_fastest(tmp_path, monkeypatch, kw):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("LBM_TUNE_CACHE", str(path))
    monkeypatch.setattr(tune.torch.cuda, "get_device_name", lambda *a, **k: "FakeGPU")
    monkeypatch.setattr(tune, "_time", lambda cfg, *a, **k: 1.0 if cfg == DEFAULT else 2.0)
    # what the cache kept before the default launch was among the candidates
    old = f"FakeGPU|128x128|{kw['prec']}|periodic,periodic|c0d0|K0|s{kw.get('scheme', 'B')}"
    path.write_text(json.dumps({old: {"config": dict(DEFAULT, kernel_variant=1, block_rows=8)}}))
    assert tune.tune(128, 128, **kw) == DEFAULT
    assert len(json.loads(path.read_text())) == 2
    key = tune._ensemble_key([dict(nx=64, ny=64)], 0, 1)
    assert key.startswith("FakeGPU|ensemble|1|") and key.endswith(f"|v{tune._VERSION}")
