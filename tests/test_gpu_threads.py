"""Samplers of different latent dimensions stepped from two host threads.

A handle belongs to one thread at a time, but different handles may run on
different threads: every launch must be right whatever the other thread
launches between its preparation and itself.  Direct launches (no graph), so
that every step prepares each of its launches again.  The draws are those of
the same sampler alone.
"""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

STEPS = 250


@pytest.mark.parametrize("path,dims,more", [
    ("mixed", (33, 128), {}),                 # persistent kernel, draw
    ("binned", (60, 128), {}),                # one CTA per row, scatter
    ("binned", (100, 128), {"tiny_max": 32}),  # tiny rows
    ("mixed", (50, 100), {"heavy_kernel": 2}),  # tensor-core Cholesky
    ("binned", (8, 128), {"hub_min": 8}),      # hubs
])
def test_two_threads(gpu_lib, path, dims, more):
    bp = gpu_lib
    ds = synth.uniform(300, 200, 4000, 8, seed=5)

    def run(K, out, errors):
        try:
            with bp.Sampler(ds.M, ds.N, ds.train_row, ds.train_col, ds.train_val, K=K, seed=K,
                            path=bp.PATH_MIXED if path == "mixed" else bp.PATH_BINNED, **more) as s:
                s.set_graph(False)
                for _ in range(STEPS):
                    s.step()
                out[K] = s.get_state()[:2]
        except Exception as ex:  # reported by the main thread
            errors.append((K, repr(ex)))

    alone, both, errors = {}, {}, []
    for K in dims:
        run(K, alone, errors)
    assert not errors, errors
    ts = [threading.Thread(target=run, args=(K, both, errors)) for K in dims]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for K in dims:
        for a, b in zip(alone[K], both[K]):
            assert np.array_equal(a, b)
