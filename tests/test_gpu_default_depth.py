"""The default chunk depth follows the form of the step, the tapered default
list does not take the estimate made for uniform ones, and a depth that was
asked for stays; none of it changes the state."""
import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture()
def make():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("depths of 152 SMs")
    from paper_1907_13415_gb300 import nlc
    sims = []

    def new(shape):
        w = wl.sphere_256().with_(shape=shape, size=0.3 * min(shape), noise=1e-3, seed=6)
        s = nlc.Simulation(wl.D3Q19, shape, w.params, precision=nlc.NLC_FP32,
                           stream=torch.cuda.current_stream().cuda_stream)
        s.set_fields(w.initial_q5())
        sims.append(s)
        return s
    yield new
    for s in sims:
        s.close()


def test_depth_by_form(make):
    s, ref = make((50, 180, 70)), make((50, 180, 70))
    assert s.chunk() == (12, False)
    s.step(2)
    s.set_persistent(3)
    assert s.chunk() == (4, False)
    s.step(3)
    s.set_persistent(0)
    assert s.chunk() == (12, False)
    s.step(2)
    ref.set_chunk(5)
    ref.step(7)
    assert np.array_equal(s.get_populations(), ref.get_populations())
    t = make((90, 67, 51))
    assert t.chunk() == (3, False)
    t.set_stencil(1)
    assert t.chunk() == (4, False)
    t.set_stencil(0)
    t.set_chunk(7)
    t.set_stencil(1)
    assert t.chunk() == (7, False)
    t.set_chunk(0)
    assert t.chunk() == (4, False)


def test_tapered_default(make):
    s = make((32, 32, 32))
    assert s.chunk() == (1, False)
    s.set_chunk(0, True)
    assert s.chunk() == (4, True)
    s.set_stencil(1)
    assert s.chunk() == (4, True)
