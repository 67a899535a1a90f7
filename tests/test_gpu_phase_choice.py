"""Which phase builds the sets, told by the launches of a growth step: the warp phase is one more. A limit of
0 that was asked for means every set by a block; a handle whose tuning was never set decides by the sets'
size and number, and for LT sets."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def growth_launches(H, graph, strategy, first, theta):
    pool = graph.pool(tag=0, roots="plain", strategy=strategy).sample(first)
    before = H.hyperim_kernel_launches()
    pool.sample(theta)
    return H.hyperim_kernel_launches() - before


@pytest.mark.parametrize("strategy,more,warps", [("paper", -1, 0), ("paper", 0, 1), ("lt", -1, 1)])
def test_phase_of_a_growth_step(strategy, more, warps):
    import paper_2406_01911_gb300 as H
    steps = 64 * torch.cuda.get_device_properties(0).multi_processor_count + more
    off = np.arange(0, 478 * 6 + 1, 6, dtype=np.int32)
    mem = np.random.default_rng(4).integers(0, 1188, size=478 * 6, dtype=np.int32)
    free, blocks, limit, tuned = (H.Graph(1188, off, mem, "wc", 0, seed=5) for _ in range(4))
    blocks.set_tuning(warp_set_limit=0)
    limit.set_tuning(warp_set_limit=128)
    assert free.tuning() == blocks.tuning()
    took = [growth_launches(H, g, strategy, 100, 100 + steps) for g in (free, blocks, limit, blocks.share())]
    assert took == [took[1] + warps, took[1], took[1] + 1, took[1]]
    # the autotuner's 0 is the handle's own choice
    tuned.set_tuning(warp_set_limit=0)
    if tuned.autotune(roots="plain", strategy=strategy, sets=64)["warp_set_limit"] == 0:
        assert growth_launches(H, tuned, strategy, 100, 100 + steps) == took[0]
