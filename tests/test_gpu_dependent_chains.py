"""Chains of reorders, traces and table updates over reused buffers, enqueued
without a synchronisation: each kernel starts while the one before it drains, and
every result is the one of the same calls made one at a time, bit for bit."""
import pytest
import torch

from paper_2506_11273_gb300 import rr
from paper_2506_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [33, 4097, 300_001, (1 << 21) - 1, (1 << 21) + 5]


def _perm(n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randperm(n, generator=g, device="cuda").to(torch.int32)


@pytest.mark.parametrize("n", SIZES)
def test_reorders_back_and_forth(n):
    g = torch.Generator("cuda").manual_seed(n)
    a = [torch.randint(-2 ** 31, 2 ** 31 - 1, (n, 4), generator=g, device="cuda", dtype=torch.int32).view(torch.float32)
         for _ in range(2)] + [torch.arange(n, device="cuda", dtype=torch.int32)]
    b = [torch.empty_like(x) for x in a]
    perms = [_perm(n, s) for s in range(3)]
    want = [x.view(torch.int32).clone() for x in a]
    for k in range(9):
        at = perms[k % 3].long()
        want = [x[at] for x in want]
    torch.cuda.synchronize()
    for k in range(9):
        rr.rr_permute(*a, perms[k % 3], *b)
        a, b = b, a
    torch.cuda.synchronize()
    for x, w in zip(a, want):
        assert torch.equal(x.view(torch.int32), w)
    assert rr.rr_device_error() == 0


@pytest.mark.parametrize("n", [33, 4097, 16_385, 300_001])
def test_bounces_over_reused_buffers(n):
    """Six bounces of three sets of rays through the same key, order, ray and table buffers; each has its own hits."""
    tris = W.scene_box_soup(seed=3)
    lo, hi = W.scene_aabb(tris)
    bvh = rr.BVH(tris)
    rays = [rr.to_device_rays(W.rays_box_soup(tris, n=n, seed=s)) for s in (1, 2, 3)]
    params = rr.key_params(rr.RR_KEY_TWO_POINT, 32, lo, hi)
    ws = rr.sort_workspace(n, 32)
    keys, perm = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    o, d = (torch.empty(n, 4, device="cuda") for _ in range(2))

    def chain(wait):
        table = rr.LengthTable(lo, hi)
        out = []
        for _ in range(2):
            for oi, di, _ in rays:
                hits, by_order = (torch.empty(n, 4, device="cuda") for _ in range(2))
                steps = [lambda: rr.rr_key_sort(oi, di, params, keys, perm, 8, ws),
                         lambda: rr.rr_trace_ex(bvh, oi, di, by_order, order=perm),
                         lambda: rr.rr_permute(oi, di, None, perm, o, d, None),
                         lambda: rr.rr_trace_accumulate(bvh, o, d, hits, table)]
                for step in steps:
                    step()
                    if wait:
                        torch.cuda.synchronize()
                out += [hits, by_order]
        torch.cuda.synchronize()
        cells = table.read()
        table.close()
        return out + [perm.clone(), o.clone(), d.clone()], cells

    want, want_cells = chain(True)
    got, cells = chain(False)
    for x, w in zip(got, want):
        assert torch.equal(x.view(torch.int32), w.view(torch.int32))
    for x, w in zip(cells, want_cells):
        assert (x == w).all()
    assert rr.rr_device_error() == 0
