"""The float64 step where the workspaces of its cell kernels are missing: the
tiled kernels take over, under a limit of device memory (NLC_ALLOC_LIMIT) and
in a stream capture that precedes the first fields.  They are held to the
oracle within the bounds of the parity tests (1e-12; float populations:
fp32_tolerance), and to each other bit for bit over chunk lists and
population offsets; what fitted without the workspaces still fits."""
import re

import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

from helpers import fp32_tolerance, perm_to_oracle, rel, run_oracle

pytestmark = pytest.mark.gpu
TILED = {"fused_lb", "fused_be"}
CELLS = {"stress", "lb", "predict", "correct"}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def workload(lattice):
    shape = (1, 21, 40) if lattice == wl.D2Q9 else (9, 11, 34)
    base = wl.disc_256() if lattice == wl.D2Q9 else wl.sphere_256()
    return base.with_(lattice=lattice, shape=shape, size=4.0, noise=1e-2, seed=5,
                      params=dict(wl.PAPER_PARAMS))


def make(w, precision, stream=None):
    import torch
    from paper_1907_13415_gb300 import nlc
    return nlc.Simulation(w.lattice, w.shape, w.params, precision=precision,
                          stream=stream or torch.cuda.current_stream().cuda_stream)


def rates(w):
    return np.linspace(0.7, 1.6, 9 if w.lattice == wl.D2Q9 else 19)


def initial(w, precision):
    s = make(w, precision)
    s.set_fields(w.initial_q5())
    data = s.save()
    s.close()
    return data


def unlimited(w, precision, data, monkeypatch):
    """Q and populations of a saved state."""
    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    s = make(w, precision)
    s.load_state(data)
    out = s.get_fields()[0], s.get_populations()
    s.close()
    return out


def least_limit(call, monkeypatch):
    """The smallest limit (context creation: to a sixteenth) at which call() fits."""
    from paper_1907_13415_gb300 import nlc
    limit = 4096
    for _ in range(400):
        monkeypatch.setenv("NLC_ALLOC_LIMIT", str(limit))
        try:
            call()
            return limit
        except nlc.NlcError as e:
            assert nlc.STATUS[e.status] == "NLC_ENOMEM"
            needs = re.findall(r"needs (\d+) bytes", str(e))
            limit = int(needs[0]) if needs else limit + limit // 16
    raise AssertionError("no limit is enough")


def loaded(w, precision, data, setup=None):
    s = make(w, precision)
    if setup:
        setup(s)
    s.load_state(data)
    return s


def kernels(s, n=1):
    from paper_1907_13415_gb300 import nlc
    nlc.nlc_set_timing(s.ctx, True)
    s.step(n)
    used = {k for k, (_, c) in nlc.nlc_get_timing(s.ctx).items() if c}
    nlc.nlc_set_timing(s.ctx, False)
    return used


SETUPS = {"bgk": lambda s, w: None, "mrt": lambda s, w: s.set_mrt(rates(w)),
          "isotropic": lambda s, w: s.set_stencil(1)}


@pytest.mark.parametrize("setup", SETUPS)
@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "fp32_qf64"])
@pytest.mark.parametrize("lattice", [wl.D2Q9, wl.D3Q19], ids=["d2q9", "d3q19"])
def test_tiled_fallback(orc, lattice, precision, setup, monkeypatch):
    w = workload(lattice)
    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    data = initial(w, precision)
    prepare = lambda s: SETUPS[setup](s, w)  # noqa: E731
    monkeypatch.setenv("NLC_ALLOC_LIMIT", str(least_limit(
        lambda: loaded(w, precision, data, prepare).close(), monkeypatch)))
    got = []
    # chunk lists no longer than the default one, for which there is room
    for deeper, taper, wide in ((0, False, "0"), (1, False, "0"), (3, False, "1"), (4, True, "0")):
        monkeypatch.setenv("NLC_POP_INDEX64", wide)
        s = loaded(w, precision, data, prepare)
        if deeper:
            s.set_chunk(s.chunk()[0] + deeper, taper)
        assert kernels(s) == TILED
        s.step(6)
        got.append(s.save())
        s.close()
    assert all(g == got[0] for g in got)
    Q, f = unlimited(w, precision, got[0], monkeypatch)
    orc.set_mrt(lattice, rates(w) if setup == "mrt" else None)
    orc.set_stencil(1 if setup == "isotropic" else 0)
    try:
        o = run_oracle(orc, w, 7)
    finally:
        orc.set_mrt(lattice, None)
        orc.set_stencil(0)
    tol = 1e-12 if precision == 0 else fp32_tolerance(7)
    assert rel(Q, o["Q"]) < tol
    assert rel(f, o["f"][perm_to_oracle(orc, lattice)]) < tol


@pytest.mark.parametrize("lattice", [wl.D2Q9, wl.D3Q19], ids=["d2q9", "d3q19"])
def test_capture_before_the_first_fields(orc, lattice):
    import torch
    w = workload(lattice)
    stream = torch.cuda.Stream()
    s = make(w, 0, stream.cuda_stream)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        s.step(2)
    s.set_fields(w.initial_q5())
    with torch.cuda.stream(stream):
        for _ in range(3):
            g.replay()
    torch.cuda.synchronize()
    o = run_oracle(orc, w, 6)
    assert rel(s.get_fields()[0], o["Q"]) < 1e-12
    assert rel(s.get_populations(), o["f"][perm_to_oracle(orc, lattice)]) < 1e-12
    s.close()


@pytest.mark.parametrize("lattice", [wl.D2Q9, wl.D3Q19], ids=["d2q9", "d3q19"])
def test_what_fitted_without_the_workspaces_still_fits(lattice, monkeypatch):
    w = workload(lattice)
    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    data = initial(w, 0)
    ref = make(w, 0)
    ref.load_state(data)
    ref.step(3)
    want = ref.get_populations()
    ref.close()
    least = least_limit(lambda: loaded(w, 0, data).close(), monkeypatch)
    n = int(np.prod(w.shape))
    read = 8 * n * (9 if lattice == wl.D2Q9 else 19)
    seen = set()
    for extra in range(0, 60):
        monkeypatch.setenv("NLC_ALLOC_LIMIT", str(least + read + 8 * n * extra))
        s = loaded(w, 0, data)
        seen.add(frozenset(kernels(s, 3)))
        assert rel(s.get_populations(), want) < 1e-12
        s.load_state(data)
        s.step(3)
        assert rel(s.get_populations(), want) < 1e-12
        s.close()
    assert seen == {frozenset(TILED), frozenset(CELLS)}


def test_a_batch_gives_back_what_it_took(monkeypatch):
    """The workspaces of the first lattice fit, those of the second do not:
    both are left to later calls."""
    import torch
    from paper_1907_13415_gb300 import nlc
    ws = [workload(wl.D2Q9).with_(shape=(1, 16, 32)), workload(wl.D2Q9).with_(shape=(1, 64, 64))]

    def batch():
        return nlc.Batch(wl.D2Q9, [w.shape for w in ws], [w.params for w in ws], precision=0,
                         stream=torch.cuda.current_stream().cuda_stream)

    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    b = batch()
    for i, w in enumerate(ws):
        b.set_fields(i, w.initial_q5())
    data = nlc.nlc_save(b.ctx)
    b.step(3)
    want = [b.get_populations(i) for i in range(2)]
    b.close()

    def load():
        c = batch()
        nlc.nlc_load(c.ctx, data)
        return c

    least = least_limit(lambda: load().close(), monkeypatch)
    read = 8 * 9 * (16 * 32 + 64 * 64)  # the populations of both lattices
    monkeypatch.setenv("NLC_ALLOC_LIMIT", str(least + read))
    b = load()
    b.step(3)
    for i in range(2):
        assert rel(b.get_populations(i), want[i]) < 1e-12
    b.close()


def test_autotune_leaves_the_cell_kernels(monkeypatch):
    from paper_1907_13415_gb300 import nlc
    monkeypatch.delenv("NLC_TUNE_CACHE", raising=False)
    w = workload(wl.D2Q9)
    Q0 = w.initial_q5()

    def fields():
        s = make(w, 0)
        s.set_fields(Q0)
        return s

    monkeypatch.setenv("NLC_ALLOC_LIMIT", str(64 + least_limit(lambda: fields().close(),
                                                              monkeypatch) + 4096))
    s = fields()
    assert kernels(s) == CELLS
    with pytest.raises(nlc.NlcError):
        s.autotune(trial_steps=2)
    assert kernels(s) == CELLS
    s.close()


def test_autotune_without_room_returns_borrowed_workspaces(monkeypatch):
    """In a context filled by load_state the saved state may take the room of
    the cell kernels' workspaces; if it does not fit even so, they come back."""
    from paper_1907_13415_gb300 import nlc
    monkeypatch.delenv("NLC_TUNE_CACHE", raising=False)
    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    w = workload(wl.D3Q19)  # the saved state is the larger of the two here
    data = initial(w, 0)
    least = least_limit(lambda: loaded(w, 0, data).close(), monkeypatch)
    word = 8 * int(np.prod(w.shape))
    results = set()
    for words in range(20, 45):
        monkeypatch.setenv("NLC_ALLOC_LIMIT", str(least + words * word))
        s = loaded(w, 0, data)
        first = kernels(s)
        try:
            s.autotune(trial_steps=2)
            tuned = True
        except nlc.NlcError as e:
            assert nlc.STATUS[e.status] == "NLC_ENOMEM"
            tuned = False
        assert kernels(s) == first
        results.add((first == CELLS, tuned))
        s.close()
    assert {(True, False), (True, True)} <= results


def test_mrt_takes_no_more_than_its_coefficients(monkeypatch):
    """With room for the coefficients the cell kernels go on with MRT, without
    it the collision is refused and BGK stays."""
    from paper_1907_13415_gb300 import nlc
    w = workload(wl.D2Q9)
    Q0, r = w.initial_q5(), rates(w)
    want = {}
    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    for mrt in (False, True):
        ref = make(w, 0)
        ref.set_fields(Q0)
        ref.set_mrt(r if mrt else None)
        ref.step(3)
        want[mrt] = ref.get_fields()[0]
        ref.close()

    def fields():
        s = make(w, 0)
        s.set_fields(Q0)
        s.get_fields()
        return s

    limit = least_limit(lambda: fields().close(), monkeypatch)
    for limit in range(limit, limit + 4096, 32):  # and the cell kernels' descriptors
        monkeypatch.setenv("NLC_ALLOC_LIMIT", str(limit))
        s = fields()
        used = kernels(s)
        s.close()
        if used == CELLS:
            break
    for extra, mrt in ((0, False), (8 * 2 * 9, True)):
        monkeypatch.setenv("NLC_ALLOC_LIMIT", str(limit + extra))
        s = fields()
        if mrt:
            s.set_mrt(r)
        else:
            with pytest.raises(nlc.NlcError):
                s.set_mrt(r)
        assert kernels(s, 3) == CELLS
        assert np.array_equal(s.get_fields()[0], want[mrt])
        s.close()
