"""The bucket sort of the tile lists at the lines of its rules, bit for bit against numpy's sort of the same
64-bit keys: depth ranges about the bin counts (fewer words than bins are binned as they are, wider ranges
by a multiplication), lists about the bins' sizing, and depth bands about the crowding limit, above which
a list goes to the radix sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sort_all(lists):
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs
    off = np.concatenate([[0], np.cumsum([len(k) for k in lists])]).astype(np.int32)
    keys = torch.tensor(np.concatenate(lists).view(np.int64), device="cuda")
    icgs.sort_tile_lists(torch.tensor(off, device="cuda"), keys)
    return [k.view(np.uint64) for k in np.split(keys.cpu().numpy(), off[1:-1])]


def _keys(rng, words):
    idx = rng.choice(5_000_000, size=len(words), replace=False).astype(np.uint64)
    return (np.asarray(words, np.uint64) << np.uint64(32)) | idx


def _check(lists):
    for k, got in zip(lists, _sort_all(lists)):
        assert np.array_equal(got, np.sort(k)), f"list of {len(k)} keys"


@pytest.mark.parametrize("n", [2, 17, 18, 128, 129, 512, 513, 1024, 1025, 2048, 2049, 4096, 4097, 8193])
def test_ranges_about_the_bin_counts(n):
    rng = np.random.default_rng(n)
    base = int(np.float32(1.7).view(np.uint32))
    lists = []
    for span in [1, 2, 255, 256, 257, 2047, 2048, 2049, 4095, 4096, 8191, 8192, 8193, 1 << 20, (1 << 30) - 1]:
        lo = base if span < 1 << 24 else 1
        words = lo + rng.integers(0, span, n)
        words[0], words[-1] = lo, lo + span - 1  # both ends of the range
        lists.append(_keys(rng, words))
    _check(lists)


@pytest.mark.parametrize("n", [40, 300, 1000, 1900, 4000, 9000])
def test_bands_about_the_crowding_limit(n):
    rng = np.random.default_rng(100 + n)
    lists = []
    for crowd in [0.02, 0.05, 0.1, 0.2, 0.4, 0.8, 1.0]:
        for width in [1, 16, 1 << 10, 1 << 16]:  # words of the band that the crowd falls in
            words = rng.integers(0x3F000000, 0x41000000, n)
            c = int(crowd * n)
            words[:c] = 0x40100000 + rng.integers(0, width, c)
            lists.append(_keys(rng, rng.permutation(words)))
    _check(lists)
