"""A wait budget of 0 (nlc_set_wait_budget): every launch of the persistent
kernel over more than one block reports the wait that ran out, however close
together its blocks arrive."""
import pytest

from paper_1907_13415_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 8, 64), (1, 64, 64)], ids=["2_blocks", "16_blocks"])
def test_every_launch_reports_it(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_13415_gb300 import nlc
    w = wl.disc_256().with_(shape=shape, size=3.0, noise=1e-3, seed=9)
    s = nlc.Simulation(w.lattice, shape, w.params, precision=nlc.NLC_FP32,
                       stream=torch.cuda.current_stream().cuda_stream)
    s.set_chunk(1, False)
    s.set_persistent(1)
    s.set_wait_budget(0)
    for _ in range(200):
        with pytest.raises(nlc.NlcError) as e:
            s.step(1)
            s.get_populations()
        assert e.value.status == -5
    s.set_wait_budget(-1)
    s.set_fields(w.initial_q5())
    s.step(3)
    assert s.observables()["nonfinite"] == 0
    s.close()
