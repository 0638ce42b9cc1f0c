"""Candidate lists of 1,025 .. 4,096 decodes where the list pass's threshold has to work:
the listed walk against the staged walk, which reads no lists, bit for bit.

Bottlenecks are set so that scores are all distinct (the threshold leaves more pairs than the
list holds), nearly all equal (pairs at the threshold in rank order), equal in blocks of
consecutive decodes (one lane's four), few below a plateau, or infinite (a bottleneck of zero;
in a chunk of few decodes the threshold itself); tight token caps send the walk past the
list to the bound.  Pools: a last chunk of 1, 4 and 100 decodes, rows that are and are not
16-byte aligned, full chunks."""
import pytest

from tests.test_gpu_listed import _assert_same, _cuda, _run, _sizes, _weights, _workload  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu



def _workload_of(D):
    """A workload of exactly D decodes: an alternating tree of 2 D instances."""
    import synth
    from tests.gpu_common import run_gpu
    spec = synth.Spec(name="lists", fanout=(1, 1, D, 2), role_rule="alternate", n_streams=3,
                      requests_per_stream=120, rate_per_s=60.0, len_median=2048.0,
                      len_clip=(16, 16384), n_roots=6, root_blocks=(1024,), n_keys=2000,
                      log2_cap=12, tables="shared", telemetry="shared", cap_tokens=60_000)
    w = synth.make_workload(spec)
    sc, x, out = run_gpu(w, cap=60_000)
    assert int(out.status.item()) == 0 and sc.D == D
    return w, sc, x, out


@pytest.mark.parametrize("D", [1025, 1028, 1124, 2048, 2049, 4096])
@pytest.mark.parametrize("scores", ["distinct", "equal", "blocks", "plateau", "infinite"])
def test_lists_of_constructed_scores(D, scores):
    w, sc, x, out = _workload_of(D)
    g = torch.Generator(device="cuda").manual_seed(D)
    UB = out.UB
    n_snap, N = UB.shape[0], UB.shape[1]
    rnd = torch.rand((n_snap, N, 1), generator=g, device="cuda")
    if scores == "distinct":
        v = 1e9 + 9e9 * rnd
    elif scores == "equal":
        v = torch.full((n_snap, N, 1), 5e9, device="cuda")
    elif scores == "blocks":
        v = 1e9 * (1 + (torch.arange(N, device="cuda") // 8 % 40)).float().view(1, N, 1).expand(n_snap, N, 1)
    elif scores == "plateau":
        v = torch.where(rnd < 0.01, 9e9 + rnd * 1e9, torch.full_like(rnd, 5e9))
    else:
        v = torch.where(rnd < 0.7, torch.zeros_like(rnd), 1e9 + 9e9 * rnd)
    UB.copy_(v.expand(n_snap, N, 4))
    UB[:, 0::2] = 2e10          # the prefills never bound a path
    x.length |= 1               # a token is always missing: no 0 x infinity
    full, rows = _sizes(x.R, D)
    for wt in (_weights(w), _weights(w, cap=3_000), _weights(w, scale_load=1e3)):
        _assert_same(_run(sc, x, out, wt, None, full), _run(sc, x, out, wt, None, rows))
