"""Prefix sharing of pools of several decode groups: known common prefixes with the leader
(chains that leave the leader's run at, before and after its end, on a block boundary or not),
leaders chosen by what the first group caches, first blocks that it does not cache, and call
sizes on both sides of the direct match.  Against the oracle's first-miss scan; every case
runs without and with a workspace (tests.test_gpu_parity._prefix_case)."""
import numpy as np
import pytest

from tests.test_gpu_parity import _prefix_case

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


@pytest.mark.parametrize("first_group", ["deepest", "shallow", "none", "shuffled"])
@pytest.mark.parametrize("D,copies", [(65, 1), (72, 60), (130, 40), (2120, 6), (2123, 6)])
def test_shared_roots(D, copies, first_group):
    """copies = 1: few enough tasks for the direct match; else sharing (more than 4,864
    (request, group) tasks).  The first group caches the roots deepest, to a shallow depth
    (every chain leaves its run at the same block), not at all, or out of order."""
    rng = np.random.default_rng(D + copies)
    roots = [_hashes(rng, 400) for _ in range(3)]
    lengths = [0, 1, 31, 127, 128, 129, 256, 300, 399, 400]
    chains = []
    for c in range(copies):
        for root in roots:
            for k in lengths:
                tail = _hashes(rng, [0, 1, 200][(c + k) % 3])
                chains.append(np.concatenate([root[:k], tail]))
    chains += [chains[5].copy(), np.zeros(0, np.uint64)]
    chains += [np.concatenate([roots[0][:200], roots[1][200:300]])]
    while copies > 1 and len(chains) * -(-D // 64) <= 4864:
        chains += chains[:1000]
    caches = []
    for d in range(D):
        depth = rng.integers(0, 401, 3)
        if d < 64:
            depth = {"deepest": np.full(3, 400 if d == 3 else 90), "shallow": np.full(3, 128),
                     "none": np.zeros(3, int), "shuffled": depth}[first_group]
        keys = np.concatenate([r[:k] for r, k in zip(roots, depth)] + [_hashes(rng, 4)])
        if d == D - 1:  # a decode that caches whole chains, tails included
            keys = np.concatenate([chains[i] for i in (2, 6, 8)])
        caches.append(rng.permutation(keys) if d < 64 and first_group == "shuffled" else keys)
    M, want, status, _ = _prefix_case(chains, [caches], D, [len(chains)])
    assert status == 0
    np.testing.assert_array_equal(M, want)


@pytest.mark.parametrize("D,steps", [(65, 3), (70, 8), (129, 13)])
def test_paths_over_several_runs(D, steps):
    """The first group's decodes cache one root ever deeper, with keys of their own between, so
    its chain is followed over `steps` runs (8 are recorded); chains leave the root before, at
    and after each run's end, for a tail or another cached chain, or end there.  D odd: request
    rows of M off the 4-byte grid."""
    rng = np.random.default_rng(D)
    root, other = _hashes(rng, 40 * steps + 40), _hashes(rng, 400)
    ends = [40 * (i + 1) for i in range(steps)]
    chains = []
    for k in sorted({e + x for e in ends for x in (-20, -1, 0, 1)} | {len(root)}):
        for tail in (np.zeros(0, np.uint64), _hashes(rng, 3), other[:50], other[50:60],
                     np.concatenate([other[:20], root[k:k + 30]])):
            chains.append(np.concatenate([root[:k], tail]))
    base = len(chains)
    while len(chains) * -(-D // 64) <= 4864:
        chains += [np.concatenate([c, _hashes(rng, 2)]) for c in chains[:base]]
    caches = []
    for d in range(D):
        if d < 64:  # deeper and deeper over the first decodes, then any depth
            depth = ends[d] if d < steps else int(rng.integers(0, ends[-1] + 1))
        else:
            depth = int(rng.integers(0, len(root) + 1))
        caches.append(np.concatenate([root[:depth], _hashes(rng, 5), other[:d % 80]]))
    M, want, status, _ = _prefix_case(chains, [caches], D, [len(chains)])
    assert status == 0
    np.testing.assert_array_equal(M, want)
