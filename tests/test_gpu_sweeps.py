"""The one-launch ternarization at the edges of its ranges: one cluster or a cooperative grid (8192 words), quarter-word
rounds, parts that start inside a row, rows off the 16-byte boundaries and tensors whose last vector is partial."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_04711_b200 import datagen as dg
from paper_1605_04711_b200 import twn
from _gpu_util import dev_f32, host_u32, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,extra", [
    (1, 15, 0), (9, 113, 64), (64, 2048, 0), (64, 2047, 0), (65, 2048, 0), (8193, 16, 0), (127, 1031, 0), (1, 131073, 0),
    (512, 2302, 0), (300, 4097, 128), (301, 4100, 0), (70001, 17, 0), (1024, 8192, 0)])
def test_codes_and_sums(rows, cols, extra):
    W = dg.draw(5, f"sweep{rows}x{cols}", rows * cols, "normal").reshape(rows, cols)
    ld = twn.ld_for(cols) + extra
    Wd, stats = dev_f32(W), twn.new_stats()
    packed = torch.full((rows, ld // 16), -1, dtype=torch.int32, device="cuda")
    ws = workspace(twn.ternarize_workspace_bytes())
    ref, codes = oracle.ternarize(W, 0.7)
    want = oracle.pack(codes.reshape(rows, cols), ld)
    for sweep in ("both", "codes"):
        if sweep == "both":
            twn.ternarize(Wd, 0.7, stats, packed, ld, None, ws)
        else:
            packed.fill_(-1)
            twn.ternarize_codes(Wd, rows, cols, stats, packed, ld, None, ws)
        st = twn.stats_to_host(stats)
        assert st["status"] == 0
        assert abs(st["delta"] - ref.delta) <= 1e-12 * ref.delta and abs(st["alpha"] - ref.alpha) <= 1e-12 * ref.alpha
        assert (st["n_neg"], st["n_zero"], st["n_pos"]) == (ref.n_neg, ref.n_zero, ref.n_pos)
        assert np.array_equal(host_u32(packed), want)


@pytest.mark.parametrize("rows,cols,offset", [
    (1, 3, 0), (9, 127, 0), (33, 129, 0), (17, 257, 0), (70, 513, 1), (70, 1023, 0), (5, 1025, 0), (3, 2049, 3), (7, 4097, 0),
    (4, 8190, 0), (3, 16385, 0), (2, 40003, 2), (3, 33024, 0)])
def test_filters(rows, cols, offset):
    """Teams of a warp and of a block, every vector count, chunked filters, matrices off the 16-byte boundaries."""
    W = dg.draw(6, f"filters{rows}x{cols}", rows * cols, "laplace").reshape(rows, cols)
    buf = torch.zeros(rows * cols + 8, dtype=torch.float32, device="cuda")
    Wd = buf[offset:offset + rows * cols].view(rows, cols)
    Wd.copy_(dev_f32(W))
    ld = twn.ld_for(cols) + (64 if rows == 7 else 0)
    stats = twn.new_stats_rows(rows)
    packed = torch.full((rows, ld // 16), -1, dtype=torch.int32, device="cuda")
    codes = torch.full((rows, cols), 7, dtype=torch.int8, device="cuda")
    twn.ternarize_rows(Wd, 0.7, stats, packed, ld, codes)
    got, words = twn.stats_rows_to_host(stats), host_u32(packed)
    for r in range(rows):
        ref, want = oracle.ternarize(W[r:r + 1], 0.7)
        assert got[r]["status"] == 0 and abs(got[r]["delta"] - ref.delta) <= 1e-12 * ref.delta
        assert abs(got[r]["alpha"] - ref.alpha) <= 1e-12 * ref.alpha
        assert (got[r]["n_neg"], got[r]["n_zero"], got[r]["n_pos"]) == (ref.n_neg, ref.n_zero, ref.n_pos)
        assert np.array_equal(words[r:r + 1], oracle.pack(want.reshape(1, cols), ld))
        assert np.array_equal(codes[r].cpu().numpy(), want.reshape(-1))


@pytest.mark.parametrize("rows,cols,offset", [(1, 1, 0), (1, 131, 0), (3, 33, 0), (31, 3784, 0), (129, 1030, 0), (64, 2048, 2),
                                              (9, 16416, 0), (300, 1027, 1), (1, 16384 * 9 + 5, 0)])
def test_signs(rows, cols, offset):
    W = dg.draw(7, f"signs{rows}x{cols}", rows * cols, "normal").reshape(rows, cols)
    W[0, 0] = -0.0
    buf = torch.zeros(rows * cols + 8, dtype=torch.float32, device="cuda")
    Wd = buf[offset:offset + rows * cols].view(rows, cols)
    Wd.copy_(dev_f32(W))
    ld = twn.ld_for_b1(cols)
    stats = twn.new_stats()
    packed = torch.full((rows, ld // 32), -1, dtype=torch.int32, device="cuda")
    twn.binarize(Wd, stats, packed, ld, workspace(twn.binarize_workspace_bytes()))
    st, (ref, codes) = twn.stats_to_host(stats), oracle.binarize(W)
    assert st["status"] == 0 and abs(st["alpha"] - ref.alpha) <= 1e-12 * ref.alpha and st["n_neg"] == int((W < 0).sum())
    assert np.array_equal(host_u32(packed), oracle.pack1(codes.reshape(rows, cols), ld))


@pytest.mark.parametrize("cols", [2 ** 32 + 1, 2 ** 32 + 4])
def test_rows_of_more_than_2_to_the_32_weights(cols):
    """Rows whose position does not fit in 32 bits and that are no whole number of words (34 GB of weights, all kept)."""
    if torch.cuda.mem_get_info()[0] < 45e9:
        pytest.skip("needs 45 GB of device memory")
    rows, used, ld = 2, (cols + 15) // 16, twn.ld_for(cols)
    W = torch.ones((rows, cols), dtype=torch.float32, device="cuda")
    stats = twn.new_stats()
    packed = torch.full((rows, ld // 16), -1, dtype=torch.int32, device="cuda")
    twn.ternarize(W, 0.7, stats, packed, ld, None, workspace(twn.ternarize_workspace_bytes()))
    st = twn.stats_to_host(stats)
    del W
    assert st["status"] == 0 and st["alpha"] == 1.0 and (st["n_neg"], st["n_zero"], st["n_pos"]) == (0, 0, rows * cols)
    whole, last = (int(oracle.pack(np.ones((1, n), dtype=np.int8), 64).view(np.int32)[0, 0]) for n in (16, cols % 16))
    assert bool((packed[:, :used - 1] == whole).all()) and bool((packed[:, used - 1] == last).all())
    assert not bool(packed[:, used:].any())
    del packed
    torch.cuda.empty_cache()
