"""The cost matrix at the edges of its tiles: pools that leave a thread column, a thread row,
a staged tile of prefill ranks or a split of them partly empty, matrices that are not
16-byte aligned, and level bottlenecks written by the same call.

C is compared bit for bit with the fp32 expression max(kv / UB_p, kv / UB_d) + L evaluated
by numpy on the bottlenecks of a call that asks for them alone."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BW, LAT = (900e9, 400e9, 200e9, 100e9), (1e-6, 3e-6, 6e-6, 10e-6)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _tiers(fanout, role):
    i = np.arange(len(role))
    f0, f1, f2, _ = fanout
    p, d = i[role == 0], i[role == 1]
    tau = np.full((len(p), len(d)), 3)
    for k, size in ((2, f0 * f1 * f2), (1, f0 * f1), (0, f0)):
        tau[(p // size)[:, None] == (d // size)[None, :]] = k
    return p, d, tau


@pytest.mark.parametrize("mode", ["links", "directed", "tiers"])
@pytest.mark.parametrize("fanout,n_decode,snaps,shift", [
    ((1, 1, 1, 2), 1, 3, 0),        # one prefill, one decode
    ((1, 1, 3, 2), 5, 2, 0),        # one prefill rank, scalar stores
    ((2, 3, 5, 9), 13, 2, 0),       # P = 257: a second staged tile of one rank
    ((1, 4, 8, 9), 32, 7, 0),       # P = 256: a full tile
    ((1, 8, 8, 17), 1024, 1, 0),    # 4 x 256 columns filled exactly
    ((1, 8, 8, 17), 1028, 1, 0),    # four decodes in a second column block
    ((3, 7, 9, 11), 2077, 1, 0),    # ragged rows over three column blocks, P = 2
    ((1, 8, 8, 40), 2048, 2, 1),    # C one float past a 16-byte boundary
])
def test_cost_matrix_tiles(fanout, n_decode, snaps, shift, mode):
    from paper_2606_03910_gb300 import netkv
    n = int(np.prod(fanout))
    rng = np.random.default_rng(n + n_decode)
    role = np.zeros(n, np.uint8)
    role[rng.permutation(n)[:n_decode]] = 1
    L = oracle.used_links(fanout) + 1
    topo = netkv.netkv_topology_create(fanout, role, BW, LAT, L)
    P, D = n - n_decode, n_decode
    rows = 4 if mode == "tiers" else L
    up, down = (torch.from_numpy(rng.uniform(0, 0.97, (snaps, rows)).astype(np.float32)).cuda()
                for _ in range(2))
    kv = 2.5e9

    def build(C, UB):
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        if mode == "links":
            netkv.netkv_oracle_build(topo, up, snaps, kv, C, UB, st)
        elif mode == "directed":
            netkv.netkv_oracle_build_directed(topo, up, down, snaps, kv, C, UB, st)
        else:
            netkv.netkv_oracle_build_tiers(topo, up, snaps, kv, C, UB, st)
        torch.cuda.synchronize()
        assert int(st.item()) == 0

    alone = torch.full((snaps, n, 4), -1.0, device="cuda")
    build(None, alone)
    UB = torch.full_like(alone, -1.0)
    flat = torch.full((snaps * P * D + shift + 1,), -1.0, device="cuda")
    C = flat[shift:shift + snaps * P * D]
    build(C, UB)
    assert torch.equal(UB, alone)
    only = torch.full((snaps * P * D,), -1.0, device="cuda")
    build(only, None)
    assert torch.equal(only, C)
    assert (flat[:shift] == -1).all() and float(flat[-1]) == -1.0  # nothing outside C
    p, d, tau = _tiers(fanout, role)
    q = np.float32(kv) / alone.cpu().numpy()  # correctly rounded fp32 quotients
    qp = np.take_along_axis(q[:, p], np.broadcast_to(tau, (snaps,) + tau.shape), 2)
    qd = np.take_along_axis(q[:, d], np.broadcast_to(tau.T, (snaps,) + tau.T.shape), 2)
    want = np.maximum(qp, qd.transpose(0, 2, 1)) + np.array(LAT, np.float32)[tau]
    np.testing.assert_array_equal(C.cpu().numpy().reshape(want.shape), want)


@pytest.mark.parametrize("mode", ["links", "tiers"])
@pytest.mark.parametrize("fanout,n_decode", [((1, 7, 11, 101), 6001),   # ragged, scalar stores
                                             ((1, 8, 8, 128), 6144)])   # 16-byte rows
def test_many_pairs_equal_the_snapshots_one_by_one(fanout, n_decode, mode):
    """Calls of 2^28 pairs and more keep more rows in flight: the same matrices as calls of one
    snapshot each."""
    from paper_2606_03910_gb300 import netkv
    n = int(np.prod(fanout))
    role = np.zeros(n, np.uint8)
    role[np.random.default_rng(n).permutation(n)[:n_decode]] = 1
    L = oracle.used_links(fanout)
    topo = netkv.netkv_topology_create(fanout, role, BW, LAT, L)
    P, D = n - n_decode, n_decode
    snaps = -(-(1 << 28) // (P * D))
    build = netkv.netkv_oracle_build if mode == "links" else netkv.netkv_oracle_build_tiers
    g = torch.Generator(device="cuda").manual_seed(5)
    util = torch.rand((snaps, L if mode == "links" else 4), generator=g, device="cuda") * 0.9
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    C = torch.empty((snaps, P, D), device="cuda")
    UB = torch.empty((snaps, n, 4), device="cuda")
    build(topo, util, snaps, 2.5e9, C, UB, st)
    one, ub = torch.empty((P, D), device="cuda"), torch.empty((n, 4), device="cuda")
    for s in range(snaps):
        build(topo, util[s].contiguous(), 1, 2.5e9, one, ub, st)
        assert torch.equal(C[s], one) and torch.equal(UB[s], ub)
    assert int(st.item()) == 0
