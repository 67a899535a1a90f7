"""Coverage with the seeds on chip takes no longer than with a flag per vertex (which more than 2,048 seeds,
repeats counted, fall back to), and counts the same."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sets,mean,k", [(20_000, 60, 100), (200_000, 60, 100), (200_000, 2, 2000), (1000, 60, 2000)])
def test_on_chip_no_slower_than_flags(sets, mean, k):
    import torch

    import paper_2406_01911_gb300 as H
    n, g = 4_000_000, torch.Generator(device="cuda").manual_seed(5)

    def rand(x):
        return torch.rand(x, generator=g, device="cuda", dtype=torch.float64)

    # most sets hold a member or two, a few hold hundreds; low ids are common
    sizes = (1.0 + 0.5 * (1.0 - rand(sets)) ** (-0.7)).clamp_(max=50.0 * mean)
    sizes = (sizes * (mean / sizes.mean())).to(torch.int64).clamp_(min=1)
    off = torch.zeros(sets + 1, device="cuda", dtype=torch.int64)
    torch.cumsum(sizes, 0, out=off[1:])
    mem = (rand(int(off[-1])) ** 3 * n).to(torch.int32).clamp_(max=n - 1)
    stratum = (rand(sets) * 16).to(torch.uint8).clamp_(max=15)
    few = (rand(k) ** 3 * n).to(torch.int32).clamp_(max=n - 1)
    many = few.repeat(2049 // k + 1)[:2049].contiguous()
    lam = {x: torch.empty(16, device="cuda", dtype=torch.int64) for x in (k, 2049)}

    def microseconds(seeds):
        ptr = [C.c_void_p(x.data_ptr()) for x in (off, mem, stratum, seeds, lam[len(seeds)])]
        best = 1e9
        for _ in range(7):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            for _ in range(50):
                assert H.lib().hyperim_coverage_noalloc(n, *ptr[:3], sets, ptr[3], len(seeds), ptr[4],
                                                        C.c_void_p(H.current_stream())) == 0
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 20)
        return best

    chip, flags = microseconds(few), microseconds(many)
    assert lam[k].tolist() == lam[2049].tolist()
    # 0.4 to 1.0 times as long; 1.4 times on a thousand sets when every SM entered the seeds eight times over
    assert chip < 1.2 * flags
