"""Steps captured in a caller's CUDA graph against settings changed after the
capture: the stencils and the collision kernels stay those of the capture,
parameters apply to the next replay.  Bit for bit against uncaptured steps."""
import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
SHAPE, SEED = (1, 12, 20), 7


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def workload():
    return wl.disc_256().with_(lattice=wl.D2Q9, shape=SHAPE, size=3.0, noise=1e-2, seed=SEED,
                               params=dict(wl.PAPER_PARAMS, gamma=2.705))


def sim(stream, precision):
    from paper_1907_13415_gb300 import nlc
    w = workload()
    s = nlc.Simulation(w.lattice, w.shape, w.params, precision=precision,
                       stream=stream.cuda_stream)
    s.set_fields(w.initial_q5())
    return s


RATES = np.linspace(0.7, 1.6, 9)
OTHER = dict(wl.PAPER_PARAMS, gamma=2.69, tau=1.2)
#: name: (before the capture, after it, what the uncaptured run has from the start)
CASES = {
    "standard_then_isotropic": (lambda s: None, lambda s: s.set_stencil(1), lambda s: None),
    "isotropic_then_standard": (lambda s: s.set_stencil(1), lambda s: s.set_stencil(0),
                                lambda s: s.set_stencil(1)),
    "bgk_then_mrt": (lambda s: None, lambda s: s.set_mrt(RATES), lambda s: None),
    "parameters": (lambda s: None, lambda s: s.set_params(OTHER), lambda s: s.set_params(OTHER)),
    "isotropic_parameters": (lambda s: s.set_stencil(1), lambda s: s.set_params(OTHER),
                             lambda s: (s.set_stencil(1), s.set_params(OTHER))),
}


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "fp32", "fp32_qf64"])
@pytest.mark.parametrize("name", CASES)
def test_replay_after_a_change(name, precision):
    import torch
    before, after, plain = CASES[name]
    stream = torch.cuda.Stream()
    a, b = sim(stream, precision), sim(stream, precision)
    before(a)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        a.step(2)
    after(a)
    with torch.cuda.stream(stream):
        for _ in range(3):
            g.replay()
    torch.cuda.synchronize()
    plain(b)
    b.step(6)
    assert np.array_equal(a.get_populations(), b.get_populations())
    assert np.array_equal(a.get_fields()[0], b.get_fields()[0])
    a.close()
    b.close()


@pytest.mark.parametrize("lattice", [wl.D2Q9, wl.D3Q19], ids=["d2q9", "d3q19"])
def test_replay_after_other_chunk_lists(lattice):
    """A captured graph keeps its chunk list, whatever lists are set later."""
    import torch
    from paper_1907_13415_gb300 import nlc
    shape = (1, 61, 70) if lattice == wl.D2Q9 else (23, 20, 40)
    base = wl.disc_256() if lattice == wl.D2Q9 else wl.sphere_256()
    w = base.with_(lattice=lattice, shape=shape, size=6.0, noise=1e-3, seed=SEED)
    stream = torch.cuda.Stream()
    out = []
    for captured in (False, True):
        s = nlc.Simulation(lattice, shape, w.params, precision=nlc.NLC_FP32,
                           stream=stream.cuda_stream)
        s.set_fields(w.initial_q5())
        if captured:
            s.set_chunk(4, True)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                s.step(2)
            for chunk in (64, 1, 3):  # shorter, longer, in between
                s.set_chunk(chunk)
                with torch.cuda.stream(stream):
                    g.replay()
                s.step(2)
        else:
            s.step(12)
        out.append((s.get_populations(), s.get_fields()[0]))
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
