"""The direct match (pools of at most 64 decodes, one index each) at the edges of its steps:
chains and cached prefixes around 128 blocks, lists that are not in chain order (blocks
looked up side by side) or change to it and back, runs that end with the index's capacity,
every mask width, warps that take several requests, and zero hashes.  Against the oracle's
first-miss scan; each case also runs with a workspace (tests.test_gpu_parity._prefix_case)."""
import numpy as np
import pytest

from tests.test_gpu_parity import _prefix_case, nk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _hashes(rng, n):
    return rng.integers(1, 2 ** 63, n, dtype=np.int64).astype(np.uint64)


EDGES = [0, 1, 2, 3, 31, 32, 33, 127, 128, 129, 130, 255, 256, 257, 383, 384, 385, 640]


@pytest.mark.parametrize("order", ["chain", "shuffled", "both", "runs of 4", "runs of 16"])
@pytest.mark.parametrize("D", [1, 8, 9, 16, 17, 32, 33, 64])
def test_step_edges(D, order):
    rng = np.random.default_rng(D)
    root = _hashes(rng, 700)
    chains = [np.concatenate([root[:k], _hashes(rng, t)]) for k in EDGES for t in (0, 1, 129)]
    caches = []
    for d in range(D):
        depth = EDGES[(7 * d + 5) % len(EDGES)]
        keys = np.concatenate([_hashes(rng, 3), root[:depth], _hashes(rng, 2)])
        if order == "shuffled" or (order == "both" and d % 2):
            keys = rng.permutation(keys)
        elif order == "both":  # in order, out of order, in order again
            keys[100:200] = rng.permutation(keys[100:200])
        elif order.startswith("runs"):
            k = int(order[8:])
            keys = np.concatenate([keys[k * i:k * i + k] for i in rng.permutation(-(-len(keys) // k))])
        caches.append(keys)
    M, want, status, _ = _prefix_case(chains, [caches], D, [len(chains)])
    assert status == 0
    np.testing.assert_array_equal(M, want)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256])
def test_run_to_the_end_of_the_index(n):
    """A list that fills the index's run array: the run ends where the array does."""
    rng = np.random.default_rng(n)
    log2_cap = max(1, int(n - 1).bit_length())
    fill = (1 << log2_cap) - n
    root = _hashes(rng, n)
    caches = [[np.concatenate([_hashes(rng, fill), root])]]
    chains = [np.concatenate([root[s:], _hashes(rng, t)]) for s in {0, n // 2, n - 1}
              for t in (0, 1, 200)]
    M, want, status, _ = _prefix_case(chains, caches, 1, [len(chains)], log2_cap=log2_cap)
    # a full table is searched to its end for an absent block, and says so
    assert status in (0, nk().NETKV_DEV_EFULL)
    np.testing.assert_array_equal(M, want)


def test_many_requests_a_warp():
    """90,000 short chains in four table sets, one of them empty: warps take several
    requests, across set boundaries."""
    rng = np.random.default_rng(3)
    sets, D = [30_001, 0, 59_990, 9], 5
    pool = [_hashes(rng, 6) for _ in range(40)]
    chains = [pool[i % 40][:i % 7] for i in rng.integers(0, 280, sum(sets))]
    caches = [[np.concatenate([p[:rng.integers(0, 7)] for p in pool]) for _ in range(D)]
              for _ in sets]
    M, want, status, _ = _prefix_case(chains, caches, D, sets)
    assert status == 0
    np.testing.assert_array_equal(M, want)


@pytest.mark.parametrize("at", [0, 1, 40, 128, 200])
@pytest.mark.parametrize("shuffled", [False, True])
def test_zero_hash(at, shuffled):
    """A zero hash in a chain is a miss; it is flagged when the scan reaches it."""
    rng = np.random.default_rng(at)
    chain = _hashes(rng, 300)
    keys = rng.permutation(chain) if shuffled else chain.copy()
    bad = chain.copy()
    bad[at] = 0
    M, _, status, _ = _prefix_case([bad, chain], [[keys, chain[:at]]], 2, [2])
    assert status == nk().NETKV_DEV_EDOMAIN
    assert M.tolist() == [[at, at], [300, at]]
    M, _, status, _ = _prefix_case([bad], [[keys[:0], chain[:max(at - 1, 0)]]], 2, [1])
    assert status == (nk().NETKV_DEV_EDOMAIN if at == 0 else 0)
    assert M.tolist() == [[0, max(at - 1, 0)]]


@pytest.mark.parametrize("at", [1, 2, 5, 40, 99])
@pytest.mark.parametrize("entry", ["other", "past the end"])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("D", [8, 64])
def test_corrupted_index(D, shuffled, entry, at):
    """A slot whose position does not hold its hash, or lies past the run array: where the scan
    looks the block up, it counts as a miss and sets EFULL, in lists in chain order and not."""
    from tests.gpu_common import host
    netkv = nk()
    rng = np.random.default_rng(at)
    chain = _hashes(rng, 100)
    keys = rng.permutation(chain) if shuffled else np.concatenate([chain[at:], chain[:at]])
    _, _, status, index = _prefix_case([chain], [[keys] * D], D, [1])
    assert status == 0
    log2_cap = netkv.index_log2_capacity(100)
    slots = index[:2 << log2_cap].view(-1, 2)
    hit = (slots[:, 0] == int(chain.view(np.int64)[at])).nonzero()
    assert hit.numel() == 1
    slot = int(hit[0, 0])
    slots[slot, 1] = (int(slots[slot, 1]) + 7) % 100 if entry == "other" else (1 << log2_cap) + 3
    M = torch.full((1, D), -1, dtype=torch.int16, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    off = torch.tensor([0, 100], device="cuda")
    netkv.netkv_prefix_match(index, D, log2_cap, 1, torch.from_numpy(chain.view(np.int64)).cuda(),
                             off, 1, None, M, st)
    # in chain order the lists wrap at `at`, so that the scan looks that block up there too
    assert host(M).tolist() == [[at] * D]
    assert int(st.item()) == netkv.NETKV_DEV_EFULL


@pytest.mark.parametrize("D", [17, 32, 33, 64])
@pytest.mark.parametrize("spread", [1, 3, 6, 7, 20, 64, 400])
def test_misses_of_many_decodes(D, spread):
    """First misses of a pool over `spread` blocks: of a few decodes, and of more than take a vote
    each, at one block or many, before, across and after the ends of 32 and 128 blocks."""
    rng = np.random.default_rng(D * 1000 + spread)
    root = _hashes(rng, 700)
    chains = [np.concatenate([root[:k], _hashes(rng, 2)]) for k in (0, 5, 31, 32, 100, 300, 700)]
    for base in (0, 27, 120):
        caches = [np.concatenate([root[:base + int(rng.integers(0, spread))], _hashes(rng, 3)])
                  for _ in range(D)]
        M, want, status, _ = _prefix_case(chains, [caches], D, [len(chains)])
        assert status == 0
        np.testing.assert_array_equal(M, want)
