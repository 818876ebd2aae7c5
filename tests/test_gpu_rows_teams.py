"""Per-filter ternarization at the edges of its teams: the last filter length that each number of vectors per thread holds and the
next one, on and off the 16-byte boundaries, few filters and many; against the rule in 64 bits."""
import pytest
import torch

from paper_1605_04711_b200 import twn

pytestmark = pytest.mark.gpu

EDGES = [*range(128, 1025, 128), *range(1536, 5121, 512), 6144, 7168, 8192]


@pytest.mark.parametrize("rows", [3, 300, 1500])
@pytest.mark.parametrize("cols", [c for e in EDGES for c in (e, e + 1)])
def test_edges(rows, cols):
    g = torch.Generator(device="cuda")
    g.manual_seed(cols)
    W = torch.randn((rows, cols), generator=g, device="cuda")
    ld = twn.ld_for(cols)
    packed = torch.full((rows, ld // 16), -1, dtype=torch.int32, device="cuda")
    stats = twn.new_stats_rows(rows)
    twn.ternarize_rows(W, 0.7, stats, packed, ld)
    mag = W.double().abs()
    delta = 0.7 * (mag.sum(1) / cols)
    # the sum of a filter is rounded cols times at most: no weight of these lies that near to its threshold, or the codes say which side
    close = (mag - delta[:, None]).abs() <= delta[:, None] * cols * 2.0 ** -53
    assert not close.any()
    keep = mag > delta[:, None]
    want = torch.where(keep, torch.sign(W), torch.zeros((), device="cuda")).to(torch.int8)
    got = torch.zeros((rows, cols), dtype=torch.int8, device="cuda")
    twn.unpack(packed, rows, cols, ld, got)
    assert torch.equal(got, want)
    if ld > (cols + 15) // 16 * 16:
        assert not packed[:, (cols + 15) // 16:].any()
    host = twn.stats_rows_to_host(stats)
    alpha = (mag * keep).sum(1) / keep.sum(1)
    for r in range(0, rows, max(1, rows // 7)):
        assert host[r]["n_pos"] == int((want[r] > 0).sum()) and host[r]["n_neg"] == int((want[r] < 0).sum())
        assert abs(host[r]["delta"] - float(delta[r])) <= cols * 2.0 ** -52 * float(delta[r])
        assert abs(host[r]["alpha"] - float(alpha[r])) <= cols * 2.0 ** -52 * float(alpha[r])
