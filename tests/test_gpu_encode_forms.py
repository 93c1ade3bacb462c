"""HCC keys where the slab test of the staged boxes changes form (needs a GB300): numbers of boxes
that the unrolled loop does not divide, both key types, rays that take the general test beside
rays that do not, and bounded beside unbounded rays."""
import numpy as np
import pytest

import oracle
from paper_2305_16652_gb300 import gen, hcc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def env():
    ctx = hcc.hcc_create(0)
    tris = gen.random_tris(3, 3000)
    bvh = gen.build_bvh(tris)
    h = hcc.hcc_bvh_upload(ctx, bvh, layout="exact")
    yield ctx, bvh, h
    hcc.hcc_bvh_destroy(h)
    hcc.hcc_destroy(ctx)


def _rays(n, seed, mixed):
    rng = np.random.default_rng(seed)
    org = np.concatenate([rng.random((n, 3)) * 1.6 - 0.3, np.full((n, 1), 1e-4)], 1).astype(np.float32)
    dir_ = np.concatenate([rng.normal(size=(n, 3)), np.full((n, 1), np.inf)], 1).astype(np.float32)
    if mixed:
        special = np.array([0.0, -0.0, 1e-42, np.inf, -np.inf, np.nan, 1e38, -3e38], np.float32)
        for a in range(3):
            dir_[rng.random(n) < 0.05, a] = rng.choice(special, 1)
            org[rng.random(n) < 0.03, a] = rng.choice(special, 1)
        for arr in (org, dir_):  # tmin and tmax: both signs, infinite, NaN
            at = rng.random(n) < 0.2
            arr[at, 3] = rng.choice(np.concatenate([special, rng.normal(size=8).astype(np.float32)]), at.sum())
    return org, dir_


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("cut_size,k", [(1, 1), (1, 32), (2, 5), (3, 3), (7, 16), (31, 31), (32, 32), (33, 33), (33, 64),
                                        (50, 49), (63, 64), (64, 64), (200, 64)])
def test_hcc_keys(env, cut_size, k, mixed):
    ctx, bvh, h = env
    n = 10_007
    org, dir_ = _rays(n, cut_size + k, mixed)
    cut = hcc.hcc_select_cut(ctx, h, cut_size, 0.125)
    try:
        ids = hcc.hcc_cut_info(cut)
        keys = torch.zeros(n, dtype=torch.int32 if k <= 32 else torch.int64, device=DEV)
        hcc.hcc_encode(ctx, "hcc", h, cut, torch.from_numpy(org).to(DEV), torch.from_numpy(dir_).to(DEV), k, keys)
        hcc.hcc_sync(ctx)
    finally:
        hcc.hcc_cut_destroy(cut)
    got = keys.cpu().numpy().view(np.uint32 if k <= 32 else np.uint64).astype(np.uint64)
    assert np.array_equal(got, oracle.encode_hcc(org, dir_, bvh.lo[ids], bvh.hi[ids], k))


@pytest.mark.parametrize("top,low,k", [(1, 1, 2), (3, 5, 8), (8, 8, 16), (5, 12, 32), (16, 16, 32), (33, 31, 64)])
def test_mlhcc_keys(env, top, low, k):
    ctx, bvh, h = env
    n = 5_003
    org, dir_ = _rays(n, top * low, True)
    cut = hcc.hcc_select_cut_ml(ctx, h, top, low)
    try:
        top_ids, low_ids, tf, lf = hcc.hcc_cut_ml_info(cut)
        keys = torch.zeros(n, dtype=torch.int32 if k <= 32 else torch.int64, device=DEV)
        hcc.hcc_encode(ctx, "mlhcc", h, cut, torch.from_numpy(org).to(DEV), torch.from_numpy(dir_).to(DEV), k, keys)
        hcc.hcc_sync(ctx)
    finally:
        hcc.hcc_cut_destroy(cut)
    got = keys.cpu().numpy().view(np.uint32 if k <= 32 else np.uint64).astype(np.uint64)
    ref = oracle.encode_mlhcc(org, dir_, tf, bvh.lo[top_ids], bvh.hi[top_ids], bvh.lo[low_ids], bvh.hi[low_ids], k)
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("k", [1, 2, 3, 5, 6, 12, 29, 30, 31, 32, 33, 36, 47, 48, 59, 60, 61, 63, 64])
def test_morton_keys(env, k):
    """Every number of bits per coordinate around the groups that are interleaved at once."""
    ctx, bvh, h = env
    n = 4_001
    org, dir_ = _rays(n, k, False)
    o, d = torch.from_numpy(org).to(DEV), torch.from_numpy(dir_).to(DEV)
    lo, hi = bvh.lo[0], bvh.hi[0]
    for method, ref in (("twopoint", oracle.encode_twopoint(org, dir_, lo, hi, k)),
                        ("origin", oracle.encode_origin(org, lo, hi, k)),
                        ("origin_dir", oracle.encode_origin_dir(org, dir_, lo, hi, k))):
        keys = torch.zeros(n, dtype=torch.int32 if k <= 32 else torch.int64, device=DEV)
        hcc.hcc_encode(ctx, method, h, None, o, d, k, keys)
        hcc.hcc_sync(ctx)
        got = keys.cpu().numpy().view(np.uint32 if k <= 32 else np.uint64).astype(np.uint64)
        assert np.array_equal(got, ref), method
