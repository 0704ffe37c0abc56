"""Launches of one frame on plans whose blocks are gridded on the tensor cores."""
import dataclasses

import numpy as np
import pytest

import epic_synth as synth
from gpu_common import assert_parity, oracle_image

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


@pytest.mark.parametrize("A,C,P,N,K,diam,bits,mix", [
    # channels enough for more than 1126 tiles of 128 cell pairs, and three of them
    (40, 600, 2, 64, 3, 18.0, 4, False), (40, 3, 2, 64, 3, 18.0, 4, False), (25, 1300, 1, 32, 3, 9.0, 4, False),
    (33, 500, 2, 64, 4, 18.0, 8, True),
    (80, 64, 2, 128, 5, 85.0, 4, False),     # row parts with padding rows
    (6, 1300, 2, 8, 3, 3.0, 8, False),
])
def test_one_sample(A, C, P, N, K, diam, bits, mix):
    cfg = synth.small_config(n_ant=A, n_chan=C, n_pol=P, grid_n=N, gcf_k=K, n_time=1, seed=A, diameter_m=diam, sigma=0.7)
    cfg = dataclasses.replace(cfg, input_bits=bits)
    if mix:
        cfg = dataclasses.replace(cfg, jones=synth.make_jones(cfg, seed=3, gain_rms=0.2, leak_rms=0.2))
    vn = synth.make_voltages(cfg)
    v = torch.from_numpy(vn).cuda()
    with E.Plan.from_config(cfg, path="dftgemm", max_time=64) as plan:
        assert plan.get_param("grid_kernel") == 4
        got = plan.image(v).cpu().numpy()
        graph = plan.image(v, graph=True).cpu().numpy()
        plan.sync()
    assert np.array_equal(got, graph)
    assert_parity(got, oracle_image(cfg, vn), "dftgemm", f"{A} elements")


def test_last_chunk_of_one_frame():
    # three chunks of four frames and one of one
    cfg = synth.small_config(n_ant=60, n_chan=300, n_pol=2, grid_n=128, gcf_k=3, n_time=13, seed=4, diameter_m=85.0)
    vn = synth.make_voltages(cfg)
    v = torch.from_numpy(vn).cuda()
    with E.Plan.from_config(cfg, path="dftgemm", max_time=16) as plan:
        plan.set_param("group", 1)
        want = plan.image(v)
        per_frame = plan.info()["scratch_bytes"] // plan.info()["time_chunk"]
        plan.set_param("chunk_mb", 1 + (4 * per_frame >> 20))
        assert plan.info()["time_chunk"] == 4
        got = plan.image(v)
        plan.sync()
    # the last frame's cells differ by FP32 rounding
    assert (got - want).norm() <= 2e-5 * want.norm()
