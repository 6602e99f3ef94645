"""Planar float32 launches of several waves, which take kernels compiled for
three blocks per SM (csrc/step_fused.cuh: launch_step), with each collision
and stencil: against the oracle within the float32 bound, and bit for bit
against a chunk list of one wave, which takes the kernels for two."""
import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

from helpers import fp32_tolerance, perm_to_oracle, rel, run_oracle

pytestmark = pytest.mark.gpu
SHAPE = (1, 205, 421)  # 14 x 26 tiles, ragged on both sides
STEPS = 5


@pytest.mark.parametrize("wide", ["0", "1"], ids=["ix32", "ix64"])
@pytest.mark.parametrize("mrt", [False, True], ids=["bgk", "mrt"])
@pytest.mark.parametrize("iso", [0, 1], ids=["standard", "isotropic"])
def test_three_blocks_per_sm(orc, iso, mrt, wide, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_13415_gb300 import nlc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    monkeypatch.setenv("NLC_POP_INDEX64", wide)
    w = wl.disc_256().with_(shape=SHAPE, size=50.0, noise=1e-2, seed=15,
                            params=dict(wl.PAPER_PARAMS))
    rates = np.linspace(0.7, 1.6, 9) if mrt else None
    out = []
    for chunk in (1, 4):
        tiles = 14 * -(-26 // chunk)
        assert (tiles > 2 * sms) == (chunk == 1)
        s = nlc.Simulation(w.lattice, SHAPE, w.params, precision=nlc.NLC_FP32,
                           stream=torch.cuda.current_stream().cuda_stream)
        s.set_chunk(chunk)
        s.set_stencil(iso)
        s.set_mrt(rates)
        s.set_fields(w.initial_q5())
        s.step(STEPS)
        out.append((s.get_populations(), s.get_fields()[0]))
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    if wide == "1":
        return
    orc.set_stencil(iso)
    orc.set_mrt(w.lattice, rates)
    try:
        o = run_oracle(orc, w, STEPS)
    finally:
        orc.set_stencil(0)
        orc.set_mrt(w.lattice, None)
    f, Q = out[0]
    assert rel(Q, o["Q"]) < fp32_tolerance(STEPS)
    assert rel(f, o["f"][perm_to_oracle(orc, w.lattice)]) < fp32_tolerance(STEPS)
