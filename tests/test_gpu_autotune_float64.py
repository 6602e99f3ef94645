"""The autotuner on float64 arithmetic, whose kernels do not use the chunk
list: the default is timed alone, kept, and not written to the cache file."""
import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "fp32_qf64"])
@pytest.mark.parametrize("lattice,shape", [(wl.D2Q9, (1, 40, 64)), (wl.D3Q19, (24, 16, 32))])
def test_nothing_to_choose(lattice, shape, precision, tmp_path, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_13415_gb300 import nlc
    path = tmp_path / "tune.json"
    monkeypatch.setenv("NLC_TUNE_CACHE", str(path))
    base = wl.disc_256() if lattice == wl.D2Q9 else wl.sphere_256()
    w = base.with_(lattice=lattice, shape=shape, size=5.0, noise=1e-3, seed=8)
    s = nlc.Simulation(lattice, shape, w.params, precision=precision,
                       stream=torch.cuda.current_stream().cuda_stream)
    default = s.chunk()
    s.set_fields(w.initial_q5())
    s.step(3)
    before = s.get_populations(), s.get_fields()[0]
    r = s.autotune(trial_steps=2)
    assert r["candidates"] == 1 and r["from_cache"] == 0 and r["trial_steps"] == 2
    assert r["best_ms"] == r["default_ms"] > 0
    assert s.chunk() == default and r["chunk"] == default[0]
    assert not path.exists()
    for a, b in zip(before, (s.get_populations(), s.get_fields()[0])):
        assert np.array_equal(a, b)
    s.close()
