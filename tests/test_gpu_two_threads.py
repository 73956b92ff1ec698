"""Handles of two threads, each on a stream of its own, that share kernels but not their launches' shared-memory
sizes: small channels stepping on chip, and sweeps with the state in shared memory.  No call fails, and the
states equal those of the same calls made by one thread."""
import threading

import numpy as np
import pytest

from paper_1310_7450_gb300 import inputs, lbnlm

pytestmark = pytest.mark.gpu


def two_threads(work):
    errors = []

    def guarded(k):
        try:
            work(k)
        except Exception as e:  # (reported by the test's thread)
            errors.append(e)

    ts = [threading.Thread(target=guarded, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


def params(seed):
    return dict(inputs.matched_params(0.9, 50.0, 0.1, 1e-3, 1e-6), rho_pert_amp=1e-3, seed=seed)


def test_steps_on_chip():
    import torch
    streams = [torch.cuda.Stream() for _ in range(2)]
    shapes, calls = [(65, 48), (160, 32)], 20000         # 35 and 74 KB of one kernel
    sims = [lbnlm.Channels(nx, ny, params(3), "f32", stream=s.cuda_stream) for (nx, ny), s in zip(shapes, streams)]
    refs = [lbnlm.Channels(nx, ny, params(3), "f32", stream=streams[0].cuda_stream) for nx, ny in shapes]
    try:
        two_threads(lambda k: [sims[k].step(8) for _ in range(calls)])
        for sim, ref in zip(sims, refs):
            for _ in range(calls):
                ref.step(8)
            (n, d), (m, e) = sim.populations()[0], ref.populations()[0]
            assert np.array_equal(n, m) and np.array_equal(d, e)
    finally:
        for s in sims + refs:
            s.close()


@pytest.mark.parametrize("prec,variant", [("f32", 1), ("f64", 1), ("f32", 0)])
def test_sweeps(prec, variant):
    import torch
    streams = [torch.cuda.Stream() for _ in range(2)]
    nys, calls = [16, 56], 300                           # one kernel, two sizes
    sims = [lbnlm.Channels(6, [ny], [params(5)], prec, stream=s.cuda_stream) for ny, s in zip(nys, streams)]
    refs = [lbnlm.Channels(6, [ny], [params(5)], prec, stream=streams[0].cuda_stream) for ny in nys]
    try:
        for s in sims + refs:
            lbnlm.lb_sweep_set_config(s.h, variant, 128, 1)

        def sweeps(k):
            for j in range(calls):  # (other arguments each time: captured again)
                sims[k].run_until_steady(-1.0, check_every=2, max_steps=2 + 2 * (j % 2))

        two_threads(sweeps)
        for sim, ref in zip(sims, refs):
            for j in range(calls):
                ref.run_until_steady(-1.0, check_every=2, max_steps=2 + 2 * (j % 2))
            (n, d), (m, e) = sim.populations()[0], ref.populations()[0]
            assert np.array_equal(n, m) and np.array_equal(d, e)
    finally:
        for s in sims + refs:
            s.close()
