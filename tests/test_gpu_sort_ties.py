"""Tile lists with few distinct depths (a flat scene seen face on, planes of equal depth): sorted bit for bit, and not
slower than by the radix passes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icgs():
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs as I
    I.load()
    return I


def _words(kind, rng, n):
    """Depth words of a list of n keys."""
    f = lambda x: np.asarray(x, np.float32).view(np.uint32)
    if kind == "one":
        return np.full(n, f(3.7))
    if kind == "two":
        return np.where(rng.random(n) < 0.5, f(2.0), f(5.0))
    if kind == "adjacent":
        return f(3.7) + rng.integers(0, 4, n).astype(np.uint32)
    if kind == "sixteen":
        return f(2.0 + rng.integers(0, 16, n) / 4.0)
    if kind == "mixed":  # one plane before a spread background
        return np.where(rng.random(n) < 0.9, f(3.7), f(2.0 + 4.0 * rng.random(n)))
    if kind == "ends":  # ties at both ends of the widest range and between
        return rng.choice(np.array([1, 2, 0x3F800000, 0x7F7FFFFF], np.uint32), n)
    raise ValueError(kind)


def _indices(kind, rng, n):
    if kind == "even":
        return rng.choice(3_000_000, n, replace=False)
    if kind == "clustered":  # runs of neighbours far apart
        start = rng.choice(np.array([0, 17, 1 << 20, 0x7FFF0000]), n)
        return np.unique(start + rng.integers(0, 4 * n, n))
    return np.arange(n) + (0x7FFFFFFF - n)  # the last ones


@pytest.mark.parametrize("kind", ["one", "two", "adjacent", "sixteen", "mixed", "ends"])
@pytest.mark.parametrize("indices", ["even", "clustered", "last"])
def test_few_depths_bit_for_bit(icgs, kind, indices):
    rng = np.random.default_rng(sum(map(ord, kind + indices)))
    lists = []
    for n in [2, 17, 18, 19, 33, 64, 127, 128, 129, 256, 700, 1024, 1025, 1500, 2048, 2049, 4096, 4097, 9000]:
        idx = rng.permutation(_indices(indices, rng, n)).astype(np.uint64)
        lists.append((_words(kind, rng, len(idx)).astype(np.uint64) << np.uint64(32)) | idx)
    off = np.concatenate([[0], np.cumsum([len(k) for k in lists])]).astype(np.int32)
    keys = torch.tensor(np.concatenate(lists).view(np.int64), device="cuda")
    icgs.sort_tile_lists(torch.tensor(off, device="cuda"), keys)
    for k, got in zip(lists, np.split(keys.cpu().numpy().view(np.uint64), off[1:-1])):
        assert np.array_equal(got, np.sort(k)), f"list of {len(k)} keys"


def _best_ms(icgs, off, keys):
    work, best = keys.clone(), float("inf")
    for _ in range(6):
        work.copy_(keys)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        icgs.sort_tile_lists(off, work)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


# How much longer than lists of spread depths: what the radix passes, which took every list before the bucket sort, need
# for lists of the kind, over what the bucket sort needs for spread ones (2e7 keys in lists of n).
@pytest.mark.parametrize("n,kind,radix", [(20, "one", 2.3), (128, "one", 1.8), (128, "adjacent", 3.4), (128, "mixed", 6.2),
                                          (256, "two", 6.8), (1000, "one", 1.9), (4096, "two", 4.3), (4096, "sixteen", 4.3)])
def test_few_depths_not_slower_than_by_radix_passes(icgs, n, kind, radix):
    rng = np.random.default_rng(n)
    count = 20_000_000 // n
    some = min(count, 64)  # as many different lists

    def lists(words):
        one = [(words(rng).astype(np.uint64) << np.uint64(32)) | rng.choice(3_000_000, n, replace=False).astype(np.uint64)
               for _ in range(some)]
        t = torch.tensor(np.stack(one).view(np.int64), device="cuda")
        return t.repeat((count + some - 1) // some, 1)[:count].contiguous().flatten()

    off = torch.arange(count + 1, dtype=torch.int32, device="cuda") * n
    spread = _best_ms(icgs, off, lists(lambda r: (2.0 + 4.0 * r.random(n)).astype(np.float32).view(np.uint32)))
    t = _best_ms(icgs, off, lists(lambda r: _words(kind, r, n)))
    print(f"{n} {kind} {t:.3f} ms, spread {spread:.3f}")
    assert t <= radix * spread


def _nested(rng, n):
    """Keys of one depth and neighbouring indices, but for one far index, one near depth and one far depth: the whole
    key's range is so wide that every split finds the others in one bin."""
    words = np.full(n, 0x40000000, np.uint64)
    idx = 1000 + np.arange(n, dtype=np.uint64)
    idx[n // 2] = 1 << 30
    words[n // 3] += 1000
    words[n // 4] += 1 << 28
    return rng.permutation((words << np.uint64(32)) | idx)


def _splits_refuse(keys, nb):
    """Whether the splits of a list of keys in nb bins leave it crowded: the rule of bucket.cuh's split_list."""
    n = len(keys)
    d, i = (keys >> np.uint64(32)).astype(object), (keys & np.uint64(0xFFFFFFFF)).astype(object)
    irange = max(i) - min(i) + 1
    z = (d - min(d)) * irange + (i - min(i))
    shift = max(0, (max(z)).bit_length() - 32)
    x, low = z >> shift, z & ((1 << shift) - 1)
    at = x * nb // (max(x) + 1)
    for _ in range(3):
        order, s0, new = np.unique(at), 0, np.zeros(n, object)
        for b in order:
            m = at == b
            c2 = 2 * int(m.sum())
            lo, hi = min(x[m]), max(x[m])
            new[m] = 2 * s0 + ((x[m] - lo) * c2 // (hi - lo + 1) if hi > lo else (low[m] * c2) >> shift)
            s0 += int(m.sum())
        at = new
        counts = np.unique(at, return_counts=True)[1]
        if int((counts * (counts - 1) // 2).sum()) <= 32 * n:
            return False
    return True


@pytest.mark.parametrize("n,bins", [(300, 4096), (1000, 4096), (1024, 4096), (1025, 4096), (2048, 4096), (2049, 8192),
                                    (4096, 8192)])
def test_what_the_splits_refuse_is_radix_sorted(icgs, n, bins):
    rng = np.random.default_rng(n)
    lists = [_nested(rng, n) for _ in range(5)] + [_nested(rng, n)[: n - 1] for _ in range(2)]
    assert all(_splits_refuse(k, bins) for k in lists[:1])
    off = np.concatenate([[0], np.cumsum([len(k) for k in lists])]).astype(np.int32)
    keys = torch.tensor(np.concatenate(lists).view(np.int64), device="cuda")
    icgs.sort_tile_lists(torch.tensor(off, device="cuda"), keys)
    for k, got in zip(lists, np.split(keys.cpu().numpy().view(np.uint64), off[1:-1])):
        assert np.array_equal(got, np.sort(k)), f"list of {len(k)} keys"
