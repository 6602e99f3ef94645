"""The float64 step kernels (csrc/step_cell.cuh) where their launches differ:
lattices of one cell block and of one cell more, several lattices in one
launch with and without the MRT collision, and steps captured in a caller's
CUDA graph, against the oracle within the float64 bound of the parity tests
(1e-12) or the uncaptured run bit for bit."""
import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

from helpers import perm_to_oracle, rel, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def small(shape, lattice, seed):
    return wl.disc_256().with_(lattice=lattice, shape=shape, size=3.0, noise=1e-2, seed=seed,
                               params=dict(wl.PAPER_PARAMS, gamma=2.705))


@pytest.mark.parametrize("lattice,shape", [(wl.D2Q9, (1, 1, 32)), (wl.D2Q9, (1, 3, 11)),
                                           (wl.D2Q9, (1, 1, 1)), (wl.D3Q19, (2, 2, 8)),
                                           (wl.D3Q19, (1, 3, 11)), (wl.D3Q19, (7, 5, 3))])
def test_block_edges(orc, lattice, shape):
    w = small(shape, lattice, 3)
    g, o = run_gpu(w, 6, precision=0), run_oracle(orc, w, 6)
    assert rel(g["Q"], o["Q"]) < 1e-12
    assert rel(g["f"], o["f"][perm_to_oracle(orc, lattice)]) < 1e-12


@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "fp32_qf64"])
def test_batch_with_and_without_mrt_equals_single_lattices(precision):
    from paper_1907_13415_gb300 import nlc
    ws = [small((1, 5, 13), wl.D2Q9, 4), small((1, 8, 8), wl.D2Q9, 5), small((1, 1, 70), wl.D2Q9, 6)]
    rates = np.linspace(0.7, 1.6, 9)
    b = nlc.Batch(wl.D2Q9, [w.shape for w in ws], [w.params for w in ws], precision=precision)
    b.set_mrt(1, rates)
    for i, w in enumerate(ws):
        b.set_fields(i, w.initial_q5())
    b.step(7)
    for i, w in enumerate(ws):
        s = nlc.Simulation(w.lattice, w.shape, w.params, precision=precision)
        if i == 1:
            s.set_mrt(rates)
        s.set_fields(w.initial_q5())
        s.step(7)
        assert np.array_equal(s.get_populations(), b.get_populations(i))
        assert np.array_equal(s.get_fields()[0], b.get_fields(i)[0])
        s.close()
    b.close()


@pytest.mark.parametrize("iso", [0, 1], ids=["standard", "isotropic"])
def test_steps_in_a_callers_capture(iso):
    import torch
    from paper_1907_13415_gb300 import nlc
    w = small((1, 12, 20), wl.D2Q9, 7)
    stream = torch.cuda.Stream()
    out = []
    for captured in (False, True):
        s = nlc.Simulation(w.lattice, w.shape, w.params, precision=0,
                           stream=stream.cuda_stream)
        s.set_fields(w.initial_q5())
        s.set_stencil(iso)
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                s.step(2)
            for _ in range(3):
                g.replay()
            torch.cuda.synchronize()
        else:
            s.step(6)
        out.append(s.get_fields())
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
