"""Keys with fused digit counting at the edges of the key kernel's 512-ray tiles
and of its persistent grid, single wavefronts and batches, against the unfused
calls and numpy's stable sort.  Integers: exact."""
import numpy as np
import pytest
import torch

from paper_2506_11273_gb300 import rr
from paper_2506_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LO, HI = np.zeros(3, np.float32), np.ones(3, np.float32)


def _rays(n, seed):
    rays = W.random_rays_in_box(n, [-0.2] * 3, [1.2] * 3, seed=seed)  # some outside the box
    o, d = rays.o_tmin.copy(), rays.d_tmax.copy()
    o[::7, 0] = np.nan
    o[1::11, 1] = np.inf
    d[2::13, :3] = 0.0
    d[3::17, 2] = -0.0
    d[5::19, 0] = 1e-38
    return torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda()


def _params(bits, layout=rr.RR_KEY_TWO_POINT):
    return rr.key_params(layout, bits, LO, HI)


@pytest.mark.parametrize("bits,radix", [(8, 4), (30, 8), (32, 8), (33, 4), (64, 8)])
@pytest.mark.parametrize("n", [1, 511, 512, 513, 456 * 512 - 1, 456 * 512 + 1])
def test_fused_matches_two_calls(n, bits, radix):
    o, d = _rays(n, n)
    p = _params(bits)
    keys, keys2 = (torch.empty(n, dtype=rr.key_dtype(bits), device="cuda") for _ in range(2))
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    rr.rr_key_sort(o, d, p, keys, perm, radix, rr.sort_workspace(n, bits, radix))
    rr.rr_compute_keys(o, d, p, keys2)
    torch.cuda.synchronize()
    assert torch.equal(keys, keys2)
    k = rr.keys_to_numpy(keys)
    assert int(k.max()) < 2 ** bits
    assert np.array_equal(rr.u32_to_numpy(perm), np.argsort(k, kind="stable").astype(np.uint32))
    assert rr.rr_device_error() == 0


@pytest.mark.parametrize("bits,radix", [(24, 8), (30, 8), (30, 4), (61, 8)])
@pytest.mark.parametrize("sizes", [(1,), (511, 0, 1), (513, 700, 3), (100, 456 * 512, 7)])
def test_batch_permutation(sizes, bits, radix):
    tris = W.scene_box_soup(seed=1, n_random=64)
    bvh = rr.BVH(tris)
    n = sum(sizes)
    o, d = _rays(n, 3)
    b = rr.Batch([(bvh, None, LO, HI, m) for m in sizes], rr.RR_KEY_AILA)
    hits = torch.empty(n, 4, device="cuda")
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    b.run(o, d, hits, rr.Batch.config(bits, radix, 128), perm)
    torch.cuda.synchronize()
    got, at = rr.u32_to_numpy(perm), 0
    for m in sizes:
        if m == 0:
            continue
        keys = torch.empty(m, dtype=rr.key_dtype(bits), device="cuda")
        rr.rr_compute_keys(o[at:at + m].contiguous(), d[at:at + m].contiguous(), _params(bits, rr.RR_KEY_AILA), keys)
        torch.cuda.synchronize()
        want = np.argsort(rr.keys_to_numpy(keys), kind="stable") + at
        assert np.array_equal(got[at:at + m], want.astype(np.uint32))
        at += m
    assert rr.rr_device_error() == 0
    b.close()
