"""Calls on a context that runs out of device memory (NLC_ALLOC_LIMIT): every
allocation in turn is the first that no longer fits, and each call either
fails with NLC_ENOMEM and leaves the state as it was, or gives the result of
an unlimited context (float32 bit for bit; float64 within 1e-12, the bound of
the parity tests, since the step may take other kernels)."""
import re

import numpy as np
import pytest

from paper_1907_13415_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def workload(lattice):
    shape = (1, 20, 40) if lattice == wl.D2Q9 else (10, 12, 34)
    base = wl.disc_256() if lattice == wl.D2Q9 else wl.sphere_256()
    return base.with_(lattice=lattice, shape=shape, size=4.0, noise=1e-2, seed=5)


def make(w, precision):
    import torch
    from paper_1907_13415_gb300 import nlc
    return nlc.Simulation(w.lattice, w.shape, w.params, precision=precision,
                          stream=torch.cuda.current_stream().cuda_stream)


def calls(sim, w, saved, adjoint):
    Q0 = w.initial_q5()

    def values(o):
        return np.array([v for k, v in sorted(o.items()) if np.ndim(v) == 0])

    out = [("set_fields", lambda: sim.set_fields(Q0)),
           ("load", lambda: sim.load_state(saved)),
           ("step", lambda: sim.step(3)),
           ("observables", lambda: values(sim.observables())),
           ("fields", lambda: np.concatenate([a.ravel() for a in sim.get_fields()])),
           ("populations", sim.get_populations),
           ("chunk", lambda: sim.set_chunk(1)),
           ("observables_1", lambda: values(sim.observables())),
           ("load_again", lambda: sim.load_state(saved)),
           ("set_mrt", lambda: sim.set_mrt(np.linspace(0.7, 1.6, 9 if w.lattice == wl.D2Q9 else 19))),
           ("step_mrt", lambda: sim.step(2)),
           ("unset_mrt", lambda: sim.set_mrt(None)),
           ("save", lambda: np.frombuffer(sim.save(), dtype=np.uint8)[64:])]
    if adjoint:
        out += [("set_fields_again", lambda: sim.set_fields(Q0)),
                ("adjoint", lambda: sim.adjoint(3.0, 1.0, 1.0, 5, 2)["dQ0"]),
                ("set_fields_third", lambda: sim.set_fields(Q0)),
                ("adjoint_longer", lambda: sim.adjoint(3.0, 1.0, 1.0, 7, 4)["dQ0"])]
    return out


def run(sim, w, saved, adjoint):
    """Results by name, each with the calls that led to the state it was taken
    on, and the bytes the calls that failed asked for."""
    from paper_1907_13415_gb300 import nlc
    res, needs, past = {}, [], ()
    for name, call in calls(sim, w, saved, adjoint):
        try:
            v = call()
        except nlc.NlcError as e:
            assert nlc.STATUS[e.status] == "NLC_ENOMEM", (name, e)
            needs += [int(m) for m in re.findall(r"needs (\d+) bytes", str(e))]
            continue
        if name.startswith(("set_fields", "load")):
            past = (name[:4],)
        elif name in ("step", "set_mrt", "step_mrt", "unset_mrt"):
            past += (name,)
        res[name] = (past, v)
    return res, needs


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "fp32", "fp32_qf64"])
@pytest.mark.parametrize("lattice", [wl.D2Q9, wl.D3Q19], ids=["d2q9", "d3q19"])
def test_every_allocation_can_be_the_one_that_fails(lattice, precision, monkeypatch):
    from paper_1907_13415_gb300 import nlc
    w = workload(lattice)
    monkeypatch.delenv("NLC_ALLOC_LIMIT", raising=False)
    sim = make(w, precision)
    sim.set_fields(w.initial_q5())
    sim.step(2)
    saved = sim.save()
    sim.close()
    sim = make(w, precision)
    want, needs = run(sim, w, saved, precision != 2)
    assert not needs
    sim.close()
    limit, walked, full = 1, 0, False
    while not full:
        monkeypatch.setenv("NLC_ALLOC_LIMIT", str(limit))
        walked += 1
        assert walked < 500
        try:
            sim = make(w, precision)
        except nlc.NlcError as e:
            assert nlc.STATUS[e.status] == "NLC_ENOMEM"
            limit = limit * 2 if limit < 4096 else limit + limit // 16
            continue
        got, needs = run(sim, w, saved, precision != 2)
        sim.close()
        full = not needs
        for name, (past, v) in got.items():
            ref = want[name][1]
            if v is None or past != want[name][0]:
                continue
            if precision == 1:
                assert np.array_equal(v, ref), (limit, name)
            elif v.dtype == np.uint8:
                assert v.shape == ref.shape
            else:
                assert np.abs(v - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max()), (limit, name)
        if not full:
            limit = min(needs)
    assert set(got) == set(want) and walked > 20
