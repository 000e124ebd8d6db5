"""Calls on a device whose memory is nearly taken: the lanes' scratch follows."""
import pytest

from paper_1302_0435_gb300 import synth

pytestmark = pytest.mark.gpu


def test_assignments_with_little_free_memory():
    """6.4 M pairs ask for 0.45 GB in one chunk; with 0.3 GB left the calls run
    in smaller chunks, with the results they have with room."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_0435_gb300 import build, d2
    build.build()
    d2.load()
    objs, cents = synth.image_like(N=100_000, K=64)
    ob = d2.bags_from_synth(objs, device="cuda:0")
    few = d2.bags_from_synth(objs.subset(range(20_000)), device="cuda:0")
    N, K = objs.count, cents.count
    lab = torch.empty(N, dtype=torch.int32, device="cuda:0")
    dist = torch.empty(N, dtype=torch.float64, device="cuda:0")
    every = torch.empty((N, K), dtype=torch.float64, device="cuda:0")

    def calls(bags):
        out = []
        d2.d2_assign(ctx, bags, lab, dist)
        d2.d2_sync(ctx)
        out += [lab.cpu(), dist.cpu()]
        d2.d2_mallows_all(ctx, bags, every, lab, dist)
        d2.d2_sync(ctx)
        return out + [lab.cpu(), dist.cpu(), every.cpu()]

    results = []
    for tight in (False, True):
        ctx = d2.Context(0)
        d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
        calls(few)  # loads the kernels
        block = None
        if tight:
            torch.cuda.empty_cache()
            free, _ = torch.cuda.mem_get_info()
            room = 300 << 20
            block = torch.empty(free - room, dtype=torch.uint8, device="cuda:0")
        results.append(calls(ob))
        del block
        ctx.close()
        torch.cuda.empty_cache()
    for a, b in zip(*results):
        assert torch.equal(a, b)
