"""The forms of the trace kernel against one another and the oracle: four lanes
to a ray (small launches and the end of large ones), one lane to a ray, and
traversal stacks deeper than their shared part.  A ray's hit does not depend on
the form that traced it, so all comparisons between forms are bit for bit."""
import numpy as np
import pytest
import torch

import hitcheck
import oracle
from paper_2506_11273_gb300 import rr
from paper_2506_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 38912 + 4099  # well above the largest launch that gets four lanes to a ray


@pytest.fixture(scope="module")
def soup():
    tris = W.scene_box_soup(seed=1)
    bvh = rr.BVH(tris)
    rays = W.rays_box_soup(tris, n=N, seed=7)
    o, d, _ = rr.to_device_rays(rays)
    return tris, bvh, rays, o, d


def _trace(bvh, o, d, **kw):
    hits = torch.full((o.shape[0], 4), -1.0, device="cuda")
    rr.rr_trace_ex(bvh, o, d, hits, **kw)
    torch.cuda.synchronize()
    return hits.view(torch.int32)


@pytest.mark.parametrize("flags", [0, rr.RR_TRACE_ANY_HIT])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 32, 33, 4097, 16383, 16384, 16385, 38911, 38912, 38913])
def test_small_launches_match_a_large_one(soup, n, flags):
    _, bvh, _, o, d = soup
    whole = _trace(bvh, o, d, flags=flags)
    assert torch.equal(_trace(bvh, o[:n].contiguous(), d[:n].contiguous(), flags=flags), whole[:n])
    order = torch.randperm(n, generator=torch.Generator().manual_seed(n)).to(torch.int32).cuda()
    assert torch.equal(_trace(bvh, o[:n].contiguous(), d[:n].contiguous(), flags=flags, order=order), whole[:n])


def test_large_launch_matches_oracle(soup):
    tris, bvh, rays, o, d = soup
    got = _trace(bvh, o, d).view(torch.float32).cpu().numpy()[:8192]
    want, info = oracle.trace_brute(tris, rays.o_tmin[:8192], rays.d_tmax[:8192])
    hitcheck.compare(tris, rays.o_tmin[:8192], rays.d_tmax[:8192], got, want, info)
    assert rr.rr_device_error() == 0


def _nested_clusters(levels):
    """Clusters of twelve triangles in planes x = 2^i, each a frame around the x axis of the size of its distance: a
    ray along the axis meets the boxes of every cluster, near to far, and descends towards the origin first."""
    rng = W.rng_for(11)
    out = []
    for i in range(levels):
        s = 2.0 ** (i - levels // 2)
        a = np.sort(rng.random(12)) * 2 * np.pi
        c = np.stack([np.full(12, s), s * 0.6 * np.cos(a), s * 0.6 * np.sin(a)], 1)
        out.append(c[:, None, :] + s * rng.uniform(-0.25, 0.25, (12, 3, 3)) * np.array([0.2, 1.0, 1.0]))
    return np.concatenate(out).reshape(-1, 9).astype(np.float32)


@pytest.mark.parametrize("n", [300, N])
def test_stack_beyond_its_shared_part(n):
    tris = _nested_clusters(64)
    bvh = rr.BVH(tris)
    assert 12 < bvh.info().depth <= 32
    rng = W.rng_for(5)
    d = np.concatenate([np.ones((n, 1)), rng.uniform(-0.8, 0.8, (n, 2))], 1)
    rays = W.make_rays(np.zeros((n, 3), np.float32), d.astype(np.float32), np.float32(0.0), np.float32(np.inf),
                       np.arange(n, dtype=np.uint32))
    o, dd, _ = rr.to_device_rays(rays)
    got = _trace(bvh, o, dd).view(torch.float32).cpu().numpy()
    m = min(n, 4096)
    want, info = oracle.trace_brute(tris, rays.o_tmin[:m], rays.d_tmax[:m])
    hitcheck.compare(tris, rays.o_tmin[:m], rays.d_tmax[:m], got[:m], want, info)
    assert rr.rr_device_error() == 0


def test_serialized_padding_survives(soup):
    """A stored BVH whose unused words are not zero comes back byte for byte."""
    tris, bvh, _, _, _ = soup
    data = bytearray(bvh.serialize())
    info = bvh.info()
    first = 64 + 80 * info.n_nodes
    for at in (first + 28, first + 44, first + 48 * info.n_tris + 32 * 5 + 24, first + 48 * info.n_tris + 32 * 5 + 28):
        data[at:at + 4] = b"\x01\x02\x03\x04"
    assert rr.BVH(serialized=bytes(data)).serialize() == bytes(data)
    assert rr.BVH(serialized=bvh.serialize()).serialize() == bvh.serialize()
