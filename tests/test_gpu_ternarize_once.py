"""Tensors that are read once (from 2^24 weights on): row lengths on and off the words, estimates of the threshold that hold,
that mark nearly every weight, and that miss; int8 codes; the same bits in a batch."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_04711_b200 import datagen as dg
from paper_1605_04711_b200 import twn
from _gpu_util import dev_f32, host_u32, kernel_launches, workspace

pytestmark = pytest.mark.gpu


def weights(rows, cols, kind):
    W = dg.draw(9, f"once{rows}x{cols}{kind}", rows * cols, "normal")
    if kind == "rows":           # filters of different scales: a wide window around the estimate
        W = (W.reshape(rows, cols) * np.linspace(0.1, 2.0, rows, dtype=np.float32)[:, None]).reshape(-1)
    elif kind == "near":         # half of the weights within 1e-4 of the threshold, 0.7 times the mean magnitude
        W = np.where(np.arange(W.size) % 2 == 0, 0.7, 1.3).astype(np.float32) * (1 + np.float32(1e-4) * W) * np.where(W < 0, -1, 1).astype(np.float32)
    elif kind == "some":         # every weight of the middle third that near, normal weights around it
        lo, hi = W.size // 3, 2 * W.size // 3
        rest = np.abs(W[:lo], dtype=np.float64).sum() + np.abs(W[hi:], dtype=np.float64).sum()
        W[lo:hi] = rest * 0.7 / (W.size - 0.7 * (hi - lo)) * (1 + 1e-4 * W[lo:hi]) * np.where(W[lo:hi] < 0, -1, 1)
    elif kind == "zeros":
        W[:] = 0.0
    elif kind == "unseen":       # large weights where no part is sampled: the estimate misses
        W[::8192] = 500.0
    return np.ascontiguousarray(W, dtype=np.float32).reshape(rows, cols)


@pytest.mark.parametrize("rows,cols,kind,extra,i8", [
    (4096, 4096, "normal", 0, False), (1, 2 ** 24 + 5, "normal", 64, True), (4099, 4111, "normal", 64, True), (4096, 4112, "rows", 0, True),
    (4096, 4100, "near", 0, False), (4096, 4096, "near", 0, True),
    (4096, 4096, "some", 0, True), (4099, 4111, "some", 0, False), (4096, 4096, "zeros", 0, True), (4097, 4099, "unseen", 0, False), (4096, 4096, "unseen", 0, True)])
def test_codes_and_sums(rows, cols, kind, extra, i8):
    W = weights(rows, cols, kind)
    ld = twn.ld_for(cols) + extra
    Wd, stats = dev_f32(W), twn.new_stats()
    packed = torch.full((rows, ld // 16), -1, dtype=torch.int32, device="cuda")
    codes8 = torch.full((rows, cols), 7, dtype=torch.int8, device="cuda") if i8 else None
    twn.ternarize(Wd, 0.7, stats, packed, ld, codes8, workspace(twn.ternarize_workspace_bytes()))
    ref, codes = oracle.ternarize(W, 0.7)
    st = twn.stats_to_host(stats)
    assert st["status"] == 0
    assert abs(st["delta"] - ref.delta) <= 1e-12 * ref.delta and abs(st["alpha"] - ref.alpha) <= 1e-12 * ref.alpha
    assert (st["n_neg"], st["n_zero"], st["n_pos"]) == (ref.n_neg, ref.n_zero, ref.n_pos)
    assert np.array_equal(host_u32(packed), oracle.pack(codes.reshape(rows, cols), ld))
    if i8:
        assert np.array_equal(codes8.cpu().numpy().reshape(-1), np.asarray(codes).reshape(-1))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_weights_are_reported(bad):
    W = dev_f32(weights(4096, 4096, "normal"))
    W[2000, 77] = bad
    stats, packed = twn.new_stats(), torch.zeros((4096, 256), dtype=torch.int32, device="cuda")
    twn.ternarize(W, 0.7, stats, packed, 4096, None, workspace(twn.ternarize_workspace_bytes()))
    assert twn.stats_to_host(stats)["status"] == -4


@pytest.mark.parametrize("kind,factor", [("normal", 0.7), ("normal", 0.0625), ("tiny", 2.0 ** -45)])
@pytest.mark.parametrize("rows,cols", [(4096, 4096), (4099, 4111)])
def test_the_coding_sweep_alone_gives_the_same_bits(rows, cols, kind, factor):
    """Codes, kept sum and scale of twn_ternarize are those of twn_ternarize_codes against the same threshold.  Where fp64 cannot
    hold the kept sum: a 1 in every 512 weights, so that a sample sees what there is, and beside it weights of 3 * 2^-52, all kept.
    A partial sum from 4 on rounds each of them up by 2^-52, so the sum depends on how many a thread adds to which partial sum."""
    if kind == "normal":
        W = dev_f32(weights(rows, cols, "normal"))
    else:
        W = torch.full((rows * cols,), 3 * 2.0 ** -52, dtype=torch.float32, device="cuda")
        W[::512] = 1.0
        W = W.view(rows, cols)
    ld = twn.ld_for(cols)
    both = []
    for call in (twn.ternarize, None):
        packed = torch.zeros((rows, ld // 16), dtype=torch.int32, device="cuda")
        if call:
            stats = twn.new_stats()
            twn.ternarize(W, factor, stats, packed, ld, None, workspace(twn.ternarize_workspace_bytes()))
        else:
            stats = both[0][0].clone()
            twn.ternarize_codes(W, rows, cols, stats, packed, ld, None, workspace(twn.ternarize_workspace_bytes()))
        both.append((stats, packed))
    assert torch.equal(both[0][0], both[1][0]) and torch.equal(both[0][1], both[1][1])
    ws = workspace(twn.ternarize_workspace_bytes())
    launches = kernel_launches(lambda: twn.ternarize(W, factor, both[0][0], both[0][1], ld, None, ws))
    assert launches == (1 if rows * cols <= factor * 2 ** 28 else 3)


def test_weights_off_the_32_byte_boundaries_and_batches():
    """The same bits alone, in a batch beside small tensors, and from a base that is aligned to 16 bytes only."""
    W = dev_f32(weights(4096, 4096, "normal"))
    buf = torch.zeros(W.numel() + 4, dtype=torch.float32, device="cuda")
    shifted = buf[4:].view(4096, 4096)
    shifted.copy_(W)
    small = dev_f32(weights(64, 800, "normal"))
    alone = []
    for w in (W, shifted, small):
        stats, packed = twn.new_stats(), torch.zeros((w.shape[0], twn.ld_for(w.shape[1]) // 16), dtype=torch.int32, device="cuda")
        twn.ternarize(w, 0.7, stats, packed, twn.ld_for(w.shape[1]), None, workspace(twn.ternarize_workspace_bytes()))
        alone.append((stats, packed))
    assert torch.equal(alone[0][0], alone[1][0]) and torch.equal(alone[0][1], alone[1][1])
    batch = [(w, w.shape[0], w.shape[1], twn.new_stats(), torch.zeros_like(a[1]), twn.ld_for(w.shape[1]), None)
             for w, a in zip((small, W, small, shifted), (alone[2], alone[0], alone[2], alone[1]))]
    twn.ternarize_batch(batch, 0.7, workspace(twn.ternarize_batch_workspace_bytes(len(batch))))
    for item, a in zip(batch, (alone[2], alone[0], alone[2], alone[1])):
        assert torch.equal(item[3], a[0]) and torch.equal(item[4], a[1])
