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
