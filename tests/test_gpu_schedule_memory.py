"""A schedule whose split rows need more memory than there is.

hub_min = 1 cuts every rating into a piece of its own, and a piece holds a
partial Gram of 39 KB at K = 128: ten million ratings ask for 390 GB.  The call
reports that, the schedule in effect stays, and the sampler goes on drawing what
it drew before, also with rows that are split.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hub", [1 << 30, 2048])
def test_schedule_out_of_memory_changes_nothing(gpu_lib, hub):
    bp = gpu_lib
    M, N, K = 4000, 2500, 128
    row = np.repeat(np.arange(M, dtype=np.int32), N)
    col = np.tile(np.arange(N, dtype=np.int32), M)
    val = np.random.default_rng(0).normal(size=M * N).astype(np.float32)
    with bp.Sampler(M, N, row, col, val, K=K, seed=2, path=bp.PATH_BINNED, hub_min=hub) as s:
        s.sample_hyper(0)
        U, V, hyper, _ = s.get_state()

        def draw():
            s.set_state(U, V, None, it=1)
            s.sweep(0)
            return s.get_state()[0]

        before, bins = draw(), s.sweep_info(0)[0]
        kept = [s.thresholds(side) for side in (0, 1)]
        with pytest.raises(bp.BpmfError):
            s.set_thresholds(0, [0, 0, 1, 0, 0])
        assert np.array_equal([s.thresholds(side) for side in (0, 1)], kept)
        assert np.array_equal(s.sweep_info(0)[0], bins)
        assert np.array_equal(draw(), before)
        s.sample_hyper(1)
        s.sweep(1)  # the other side shares the pieces' memory
        s.step()
