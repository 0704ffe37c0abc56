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


def test_channels_of_small_gains_are_as_accurate_as_with_single_precision_gridding():
    # gains of one in one channel and of 1e-5 in another: the split's absolute floor of 2^-25 is 1e-3 of a sample there
    cfg = synth.small_config(n_ant=60, n_chan=2, n_pol=2, grid_n=64, gcf_k=4, n_time=24, seed=7, diameter_m=18.0, sigma=0.8)
    cfg.jones = synth.make_jones(cfg, seed=3, gain_rms=0.2, leak_rms=0.2)
    cfg.jones[1] *= 1e-5
    v = synth.make_voltages(cfg)
    ref = oracle.image_cfg(cfg, v)
    err = {}
    with E.Plan.from_config(cfg, path="dftgemm") as plan:
        for kernel in (None, 1):                  # the plan's choice, then sums in FP32
            if kernel:
                plan.set_param("grid_kernel", kernel)
            got = plan.image(torch.from_numpy(v).cuda()).cpu().numpy()
            plan.sync()
            err[kernel] = [np.linalg.norm(got[c] - ref[c]) / np.linalg.norm(ref[c]) for c in range(2)]
    for c in range(2):
        assert err[None][c] <= 1.05 * err[1][c], (c, err)
