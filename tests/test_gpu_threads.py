"""Contexts made, used and destroyed by several host threads at once, each on its own
stream: while one thread records its step as a graph, the others create and destroy
contexts and read counters.  Every result equals that of the same calls made one
thread after another."""
import threading

import numpy as np
import pytest

from paper_1909_07439_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = {1: 2500, 2: 20000, 3: 9000, 4: 60000}


def _job(seed, out, errors):
    try:
        from paper_1909_07439_gb300 import DeviceState, native
        torch.cuda.set_device(0)
        w = inputs.unit_sphere(SIZES[seed], seed=seed)
        with torch.cuda.stream(torch.cuda.Stream()):
            ctx = native.sph_create(w.n, 0)
            p = native.sph_params_default(n_group=8 if seed % 2 else 32)
            s = DeviceState.from_arrays(w.pos, w.vel, w.h)
            dt = torch.full((1,), 1e-5, device="cuda")
            time = torch.zeros(1, dtype=torch.float64, device="cuda")
            native.sph_build_tree(ctx, s.c, p)
            native.sph_density(ctx, s.c, p)
            native.sph_force(ctx, s.c, p)
            for _ in range(5):
                native.sph_step(ctx, s.c, p, dt, time)
            native.sph_get_stats(ctx)
            native.sph_sync(ctx)
            out[seed] = {f: s.numpy(f).copy() for f in ("pos", "vel", "h", "rho", "acc", "perm")}
            native.sph_destroy(ctx)
    except Exception as e:  # a thread's exception would be lost
        errors.append(repr(e))


def test_threads_with_contexts_of_their_own():
    from paper_1909_07439_gb300 import build, native
    build.build()
    native.load()
    want, errors = {}, []
    for k in SIZES:
        _job(k, want, errors)
    assert not errors and set(want) == set(SIZES)
    for _ in range(4):
        got = {}
        threads = [threading.Thread(target=_job, args=(k, got, errors)) for k in SIZES]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors
        for k in SIZES:
            for f, a in want[k].items():
                assert np.array_equal(got[k][f], a), (k, f)
