"""The cache index that netkv_cache_build lays out, against a plain numpy index: every
distinct hash once, found by linear probing from its home slot, at the run position of its
first appearance in the lists, with the mask of the decodes that list it, and zeros past
the last run position.  The cases reach the edges of the build's passes: lists around the
256 elements of a count, mask widths of 1, 2, 4 and 8 bytes, lists too long for the bitmap
and tables too full for the counts (both built by one block per index).  Calls on few lists of
up to 2^13 slots, and on many indices of up to 2^14, are built by one block per index too: the
edges of the passes are reached with 17 decodes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U64 = np.uint64
GROUP = 64


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _hashes(rng, n):
    return rng.integers(1, 2 ** 64, n, dtype=U64)


def _prefix_lists(seed, D, n, roots=3):
    """Lists as caches are filled: prefixes of shared roots, then a decode's own blocks."""
    rng = np.random.default_rng(seed)
    root = [_hashes(rng, n) for _ in range(roots)]
    return [np.concatenate([r[:rng.integers(0, n + 1)] for r in root] + [_hashes(rng, 1 + d % 5)])
            for d in range(D)]


def _repeats(seed, T, distinct):
    rng = np.random.default_rng(seed)
    h = _hashes(rng, distinct)
    return [np.concatenate([h, h[rng.integers(0, distinct, T - distinct)]])]


def _among(keys, D):
    """One list among D - 1 empty ones."""
    return [[]] * (D // 2) + [keys] + [[]] * (D - 1 - D // 2)


CASES = {
    "one key, two slots": ([[5]], 1, 1, "ranked"),
    "no key": ([[], []], 2, 4, "ranked"),
    "255 elements": ([np.arange(1, 256)], 1, 10, "ranked"),
    "256 elements": ([np.arange(1, 257)], 1, 10, "ranked"),
    "257 elements": ([np.arange(1, 258)], 1, 10, "ranked"),
    "8 decodes": (_prefix_lists(1, 8, 300), 8, 12, "ranked"),
    "9 decodes": (_prefix_lists(2, 9, 300), 9, 12, "ranked"),
    "17 decodes": (_prefix_lists(3, 17, 100), 17, 11, "ranked"),
    "64 decodes": (_prefix_lists(4, 64, 500), 64, 13, "ranked"),
    "65 decodes": (_prefix_lists(5, 65, 500), 65, 13, "ranked"),
    "3 sets of 130 decodes": (_prefix_lists(6, 390, 90), 130, 11, "ranked"),
    "one long list": ([_hashes(np.random.default_rng(7), 70_000)], 1, 18, "ranked"),
    "bitmap filled": (_repeats(8, 8 * 1024, 100), 1, 10, "ranked"),
    "bitmap too small": (_repeats(9, 8 * 1024 + 1, 100), 1, 10, "any"),
    "counts fill the keys": ([np.arange(1, 1022)], 1, 10, "ranked"),  # 2 * 1021 + 5 words of 2,048
    "counts past the keys": ([np.arange(1, 1023)], 1, 10, "any"),     # 2 * 1022 + 5
    "full table": ([np.arange(1, 1025)], 1, 10, "any"),
    # the passes at the same edges: 17 lists of one index are too many for one block
    "17: 255 elements": (_among(np.arange(1, 256), 17), 17, 10, "ranked"),
    "17: 256 elements": (_among(np.arange(1, 257), 17), 17, 10, "ranked"),
    "17: 257 elements": (_among(np.arange(1, 258), 17), 17, 10, "ranked"),
    "17: bitmap filled": (_among(_repeats(8, 32 * 1024, 100)[0], 17), 17, 10, "ranked"),
    "17: bitmap too small": (_among(_repeats(9, 32 * 1024 + 1, 100)[0], 17), 17, 10, "ranked"),
    "17: counts fill the keys": (_among(np.arange(1, 1022), 17), 17, 10, "ranked"),
    "17: counts past the keys": (_among(np.arange(1, 1023), 17), 17, 10, "any"),
    "17: full table": (_among(np.arange(1, 1025), 17), 17, 10, "any"),
    # around the rule
    "12 decodes of 2^13": (_prefix_lists(10, 12, 900), 12, 13, "ranked"),
    "12 decodes of 2^14": (_prefix_lists(11, 12, 900), 12, 14, "ranked"),
    "80 sets of 12 of 2^14": (_prefix_lists(18, 960, 20), 12, 14, "ranked"),
    "80 sets of 12 of 2^15": (_prefix_lists(19, 960, 20), 12, 15, "ranked"),
    "16 decodes of 2^11": (_prefix_lists(16, 16, 200), 16, 11, "ranked"),
    "16 decodes of 2^12": (_prefix_lists(17, 16, 200), 16, 12, "ranked"),
    "300 sets of 3": (_prefix_lists(12, 900, 60), 3, 9, "ranked"),
    "300 sets of 13": (_prefix_lists(13, 3900, 30), 13, 10, "ranked"),
    "80 sets of 33": (_prefix_lists(14, 2640, 20), 33, 11, "ranked"),
    "repeats in a chunk": ([_repeats(15, 3000, 700)[0][::-1], _repeats(15, 3000, 700)[0]], 2, 11,
                           "ranked"),
}


@pytest.mark.parametrize("name", CASES)
def test_index_layout(name):
    from paper_2606_03910_gb300 import netkv
    lists, D, log2_cap, order = CASES[name]
    lists = [np.asarray(x, dtype=U64) for x in lists]
    n_sets = len(lists) // D
    off = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    keys = np.concatenate(lists) if off[-1] else np.zeros(1, U64)
    nbytes = netkv.netkv_cache_index_bytes(n_sets, D, log2_cap)
    guard = 64
    buf = torch.full((nbytes // 8 + guard,), -1, dtype=torch.int64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    netkv.netkv_cache_build(buf, n_sets, D, log2_cap, torch.from_numpy(keys.view(np.int64)).cuda(),
                            torch.from_numpy(off).cuda(), st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    raw = buf.cpu().numpy()
    assert (raw[nbytes // 8:] == -1).all()
    n_groups = -(-D // GROUP)
    cap, stride = 1 << log2_cap, nbytes // (n_sets * n_groups)
    width = next(w for w in (1, 2, 4, 8) if 8 * w >= min(D, GROUP))
    for g in range(n_sets):
        for q in range(n_groups):
            rank, bits = {}, {}
            for d in range(q * GROUP, min(D, (q + 1) * GROUP)):
                for h in lists[g * D + d].tolist():
                    rank.setdefault(h, len(rank))
                    bits[h] = bits.get(h, 0) | 1 << (d - q * GROUP)
            idx = raw.view(np.uint8)[(g * n_groups + q) * stride:][:stride]
            slots = idx[:16 * cap].view(U64).reshape(cap, 2)
            runs = idx[16 * cap:24 * cap].view(U64)
            masks = idx[24 * cap:(24 + width) * cap].view("u%d" % width)
            used = slots[:, 0] != 0
            assert sorted(slots[used, 0].tolist()) == sorted(rank)
            n = len(rank)
            assert not runs[n:].any() and not masks[n:].any() and not slots[~used, 1].any()
            for s in np.flatnonzero(used):
                h, pos = int(slots[s, 0]), int(slots[s, 1])
                assert pos == rank[h] if order == "ranked" else pos < n
                assert int(runs[pos]) == h and int(masks[pos]) == bits[h]
                i = (h * 0x9E3779B97F4A7C15 % 2 ** 64) >> (64 - log2_cap)
                while i != s:
                    assert used[i]
                    i = (i + 1) % cap


def test_bad_lists_are_flagged():
    """A zero key (EDOMAIN), a list that ends before it begins (ERANGE, skipped) and more
    distinct keys than slots (EFULL); the other lists are indexed."""
    from paper_2606_03910_gb300 import netkv

    def build(keys, off, D, log2_cap):
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        buf = torch.empty(netkv.netkv_cache_index_bytes(1, D, log2_cap) // 8, dtype=torch.int64,
                          device="cuda")
        netkv.netkv_cache_build(buf, 1, D, log2_cap, torch.tensor(keys, device="cuda"),
                                torch.tensor(off, device="cuda"), st)
        torch.cuda.synchronize()
        slots = buf.cpu().numpy()[:2 << log2_cap].reshape(-1, 2)
        return int(st.item()), sorted(slots[slots[:, 0] != 0, 0].tolist())

    assert build([1, 0, 2, 3], [0, 3, 4], 2, 4) == (netkv.NETKV_DEV_EDOMAIN, [1, 2, 3])
    assert build([1, 2, 3, 4], [0, 3, 1, 4], 3, 4) == (netkv.NETKV_DEV_ERANGE, [1, 2, 3, 4])
    status, kept = build(list(range(1, 40)), [0, 39], 1, 5)
    assert status == netkv.NETKV_DEV_EFULL and len(kept) == 32
