"""Contexts on streams of the caller's: steps are recorded without touching the caller's stream, so it may be
shared by several contexts and threads and by other work, and may be the legacy default stream."""
import threading

import numpy as np
import pytest

import synthetic as syn
from gpu_common import engine, model

pytestmark = pytest.mark.gpu

LEGACY, PER_THREAD = 1, 2   # cudaStreamLegacy, cudaStreamPerThread


def _same(a, b):
    assert a.keys() == b.keys()
    for k in a:
        np.testing.assert_array_equal(np.asarray(a[k]), np.asarray(b[k]), err_msg=k)


def _eager(eng, blob, sy):
    with eng.Potential(64, T=2, n_species=2, params=blob) as pot:
        pot.profile(True)
        return pot.compute(sy.species, sy.positions, sy.cell, energies=True)


@pytest.mark.parametrize("stream", [LEGACY, PER_THREAD])
def test_special_streams(stream):
    eng = engine()
    sy = syn.water_box(60, seed=1)
    _, blob = model(64, 2, 2, seed=3, bias=0.1)
    want = _eager(eng, blob, sy)
    with eng.Potential(64, T=2, n_species=2, params=blob, stream=stream) as pot:
        for _ in range(5):
            _same(pot.compute(sy.species, sy.positions, sy.cell, energies=True), want)


def test_one_stream_for_several_threads():
    """Two contexts and a server recording and replaying, and plain work beside them, all on one stream."""
    import torch
    eng = engine()
    _, blob = model(64, 2, 2, seed=3, bias=0.1)
    systems = [syn.water_box(60, seed=1), syn.water_box(70, seed=2)]
    want = [_eager(eng, blob, sy) for sy in systems]
    vel = syn.maxwell_boltzmann(systems[0].masses, 300.0, seed=1)
    sy0 = systems[0]

    def serve(stream):
        srv = eng.Server(64, blob, T=2, n_species=2, dt=0.5, stream=stream)
        rid = srv.submit(sy0.species, sy0.masses, sy0.positions, vel, sy0.cell, 12, skin=1.0)
        for _ in range(14):
            srv.step()
        got = srv.poll(rid)
        srv.close()
        return got["epot"]

    epot = serve(None)
    stream = torch.cuda.Stream()
    failures, done = [], threading.Event()

    def guarded(f):
        def go():
            try:
                f()
            except BaseException as e:   # reported by the main thread
                failures.append(e)
        return go

    def calls(k):
        with eng.Potential(64, T=2, n_species=2, params=blob, stream=stream.cuda_stream) as pot:
            for _ in range(30):
                pot.load_params(blob)   # drops the recordings
                for _ in range(4):
                    _same(pot.compute(systems[k].species, systems[k].positions, systems[k].cell, energies=True), want[k])

    def serves():
        for _ in range(8):
            np.testing.assert_array_equal(serve(stream.cuda_stream), epot)

    def other():
        with torch.cuda.stream(stream):
            a = torch.arange(1000, device="cuda", dtype=torch.float64)
            total = torch.zeros((), device="cuda", dtype=torch.float64)
            n = 0
            while not done.is_set():
                total += a.sum()
                n += 1
                assert float(total) == n * 499500.0

    workers = [threading.Thread(target=guarded(f)) for f in (lambda: calls(0), lambda: calls(1), serves)]
    beside = threading.Thread(target=guarded(other))
    for t in (*workers, beside):
        t.start()
    for t in workers:
        t.join()
    done.set()
    beside.join()
    assert not failures, failures
