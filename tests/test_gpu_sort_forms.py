"""The sort's forms by size and key width (needs a GB300): one cluster launch up to 65,536
keys, digit passes over small and large tiles above, and for keys above 32 bits wide passes
that hand over to 32-bit pairs, with any of the passes skipped."""
import numpy as np
import pytest

import oracle
from paper_2305_16652_gb300 import hcc
from test_gpu_parity import gpu_sort

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hcc.hcc_create(0)
    yield c
    hcc.hcc_destroy(c)


@pytest.mark.parametrize("n", [1023, 4095, 4096, 4097, 8193, 16385, 32769, 61441, 65535, 65536, 65537, 450_000, 450_001])
@pytest.mark.parametrize("k", [3, 9, 32, 33, 47, 64])
def test_sizes_where_the_form_changes(ctx, n, k):
    rng = np.random.default_rng(n + k)
    keys = rng.integers(0, 1 << min(k, 63), n, dtype=np.uint64) << np.uint64(k - min(k, 63))
    keys[rng.random(n) < 0.3] = keys[0]  # a digit that dominates
    assert np.array_equal(gpu_sort(ctx, keys, k), oracle.stable_sort(keys))


@pytest.mark.parametrize("n", [30_001, 70_001, 460_001])
@pytest.mark.parametrize("bytes_", ["0", "3", "4", "7", "01", "04", "34", "47", "12", "037", "014567", "01234567", ""])
def test_any_digits_of_64_bit_keys_may_be_equal(ctx, n, bytes_):
    """Only the listed bytes of the keys vary: the passes over the others are skipped."""
    rng = np.random.default_rng(len(bytes_) * 1000 + n)
    keys = np.full(n, 0x1122334455667788, np.uint64)
    for b in bytes_:
        shift = np.uint64(8 * int(b))
        keys &= ~(np.uint64(255) << shift)
        keys |= rng.integers(0, 256, n, dtype=np.uint64) << shift
    assert np.array_equal(gpu_sort(ctx, keys, 64), oracle.stable_sort(keys))


@pytest.mark.parametrize("k", [32, 48, 64])
@pytest.mark.parametrize("reserved,n", [(450_001, 450_000), (460_000, 450_000), (460_000, 420_000), (480_000, 430_000)])
def test_reserved_scratch_covers_smaller_sorts(k, reserved, n):
    """The tiles are smaller at 450,000 keys and take more scratch than at somewhat more: a capture, which
    cannot allocate, of a sort below the reserved size."""
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << min(k, 63), n, dtype=np.uint64)
    dev = torch.from_numpy(keys.astype(np.uint32).view(np.int32) if k <= 32 else keys.view(np.int64)).to("cuda:0")
    perm = torch.empty(n, dtype=torch.int32, device="cuda:0")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    c = hcc.hcc_create(0, stream)
    try:
        hcc.hcc_reserve(c, reserved, k)
        hcc.hcc_graph_begin(c)
        try:
            hcc.hcc_sort(c, dev, k, n, perm)
        finally:
            graph = hcc.hcc_graph_end(c)
        hcc.hcc_graph_launch(c, graph)
        hcc.hcc_sync(c)
        assert np.array_equal(perm.cpu().numpy().view(np.uint32), oracle.stable_sort(keys))
        hcc.hcc_graph_destroy(graph)
    finally:
        hcc.hcc_destroy(c)
