"""A waiting host bounce stores its hits straight into page-locked buffers: the same
bytes as through a pageable buffer, and after an earlier submission's download into
the same buffer.  Bit-exact: the kernels and their inputs are the same."""
import numpy as np
import pytest
import torch

from paper_2506_11273_gb300 import rr
from paper_2506_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("payload", [True, False])
@pytest.mark.parametrize("n", [1, 33, 16384, 16385, 300001])
def test_direct_hits_match_staged(n, payload):
    tris = W.scene_box_soup(seed=2)
    lo, hi = W.scene_aabb(tris)
    bvh = rr.BVH(tris)
    pipe = rr.Pipeline(bvh, 300001, rr.key_params(rr.RR_KEY_TWO_POINT, 32, lo, hi), radix_bits=8)
    first, r = W.rays_box_soup(tris, n=300001, seed=3), W.rays_box_soup(tris, n=n, seed=4)

    def pinned(rays):
        return [torch.from_numpy(a).pin_memory() for a in (rays.o_tmin, rays.d_tmax, rays.payload.view(np.int32))]

    want, want_pay = np.zeros((n, 4), np.float32), np.zeros(n, np.int32)
    pipe.run_host(r.o_tmin, r.d_tmax, r.payload, want, want_pay)
    hits = torch.full((300001 + 1, 4), -7.0).pin_memory()
    pay, first_pay = torch.zeros(n, dtype=torch.int32).pin_memory(), torch.zeros(300001, dtype=torch.int32).pin_memory()
    (o1, d1, p1), (o, d, p) = pinned(first), pinned(r)
    for earlier in (False, True):
        hits.fill_(-7.0)
        if earlier:  # not waited for: its download into the same buffer comes first
            pipe.submit_host(o1, d1, p1, hits, first_pay)
        pipe.run_host(o, d, p if payload else None, hits, pay if payload else None)
        assert np.array_equal(hits[:n].numpy().view(np.uint32), want.view(np.uint32))
        assert earlier or (hits[n:] == -7.0).all()
        assert not payload or np.array_equal(pay.numpy(), want_pay)
    assert rr.rr_device_error() == 0
    pipe.close()


def test_direct_hits_wait_for_downloads_before_a_failed_submission():
    """A submission still downloading, one that fails at its first launch, then a waiting bounce whose page-locked hits
    lie at the end of the first one's: the last one's hits stay."""
    big, n = 2_000_000, 33
    tris = W.scene_box_soup(seed=2)
    lo, hi = W.scene_aabb(tris)
    bvh = rr.BVH(tris)
    pipe = rr.Pipeline(bvh, big, rr.key_params(rr.RR_KEY_TWO_POINT, 32, lo, hi), radix_bits=8)
    first, r = W.rays_box_soup(tris, n=big, seed=3), W.rays_box_soup(tris, n=n, seed=4)
    o1, d1, o, d = [torch.from_numpy(a).pin_memory() for a in (first.o_tmin, first.d_tmax, r.o_tmin, r.d_tmax)]
    want = np.zeros((n, 4), np.float32)
    pipe.run_host(r.o_tmin, r.d_tmax, None, want, None)
    hits, other = torch.full((big, 4), -7.0).pin_memory(), torch.zeros(n, 4).pin_memory()
    for _ in range(3):
        hits.fill_(-7.0)
        pipe.submit_host(o1, d1, None, hits, None)
        rr.rr_fault_inject("launch@1")
        with pytest.raises(rr.RRError):
            pipe.submit_host(o, d, None, other, None)
        rr.rr_fault_inject(None)
        pipe.run_host(o, d, None, hits[big - n:], None)
        assert np.array_equal(hits[big - n:].numpy().view(np.uint32), want.view(np.uint32))
        assert not (hits[:big - n] == -7.0).any()
    assert rr.rr_device_error() == 0
    pipe.close()
