"""Groups of copies in one launch: sizes around the 16-byte unit, the chunk of each form and
the 32 buffers of a launch, host and device memory, and bad groups refused as a whole."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [0, 1, 15, 16, 17, 4096, 512 * 16 - 1, 512 * 16, 512 * 16 + 1, 2048 * 16 + 33]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("repeat,large", [(1, 0), (4, 0), (1, 100_000_019)])
@pytest.mark.parametrize("to_host", [False, True])
def test_copy_group(repeat, large, to_host):
    from paper_2606_03910_gb300 import netkv
    sizes = SIZES * repeat + ([large] if large else [])
    g = torch.Generator().manual_seed(3)
    src = [torch.randint(0, 256, (n + 16,), dtype=torch.uint8, generator=g).pin_memory() for n in sizes]
    dst = [torch.full((n + 16,), 7, dtype=torch.uint8, device="cuda") for n in sizes]
    if to_host:
        src, dst = [s.cuda() for s in src], [d.cpu().pin_memory() for d in dst]
    torch.cuda.synchronize()
    netkv.netkv_copy_group_async([(d, s, n) for d, s, n in zip(dst, src, sizes)])
    torch.cuda.synchronize()
    for d, s, n in zip(dst, src, sizes):
        assert torch.equal(d[:n].cpu(), s[:n].cpu())
        assert (d[n:] == 7).all()


def test_bad_groups_copy_nothing():
    from paper_2606_03910_gb300 import netkv
    s = torch.ones(64, dtype=torch.uint8, device="cuda")
    d = torch.zeros(64, dtype=torch.uint8, device="cuda")
    netkv.netkv_copy_group_async([])
    for bad in ((d[1:], s, 16), (d, s[1:], 16), (None, s, 16), (d, None, 16), (d, s, 1 << 40)):
        with pytest.raises(netkv.NetKVError) as e:
            netkv.netkv_copy_group_async([(d, s, 32), bad])
        assert e.value.code == netkv.NETKV_EINVAL
    torch.cuda.synchronize()
    assert not d.any()
