"""Polarisation mixing with matrices at the ends of the range that the tensor-core gridding kernel splits into FP16 parts."""
import numpy as np
import pytest

import epic_synth as synth
import oracle
from gpu_common import assert_parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402

CELL = 0.5 * 299792458.0 / 120e6


def test_largest_matrices_with_the_largest_samples_stay_finite():
    # real and imaginary parts of 128 times samples of -128: a mixed part is 4 x 2^14, just above FP16's range, while
    # grid cells (weights exp(-4) at half a cell) stay far below it
    cfg = synth.small_config(n_ant=2, n_chan=1, n_pol=2, grid_n=32, gcf_k=2, n_time=16, seed=1, sigma=0.25)
    cfg.pos_m = np.array([[-2.5, -2.5], [2.5, 2.5]]) * CELL
    cfg.input_bits = 8
    cfg.jones = np.full((1, 2, 2, 2), 128.0 + 128.0j, np.complex64)
    v = np.full((16, 1, 2, 2, 2), 0x80, np.uint8)
    ref = oracle.image_cfg(cfg, v)
    with E.Plan.from_config(cfg, path="dftgemm") as plan:
        got = plan.image(torch.from_numpy(v).cuda()).cpu().numpy()
        plan.sync()
    assert_parity(got, ref, "dftgemm", "largest mixing matrices")
