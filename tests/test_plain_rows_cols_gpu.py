"""The plain path's two kernels (gridded row FFTs of the box, column FFTs with products) at their edges."""
import dataclasses

import numpy as np
import pytest

import epic_synth as synth
from gpu_common import assert_parity, oracle_image

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402

CASES = [
    # A, C, P, N, K, T, diameter, bits, sub, mixing, chunk
    (20, 3, 2, 8, 2, 9, 3.0, 4, 0, False, 1),       # smallest grid: one column tile
    (20, 2, 1, 16, 3, 7, 4.5, 8, 0, False, 1),      # odd number of frames: the last block holds one
    (30, 1, 2, 64, 5, 67, 17.0, 4, 0, False, 1),    # one channel: slices of the frames, partial sums
    (30, 1, 1, 128, 3, 45, 34.0, 4, 0, False, 1),   # ... and several chunks of them
    (30, 2, 2, 128, 7, 12, 136.0, 8, 3, True, 1),   # a box wider than the grid's padding, intervals
    (25, 1, 2, 256, 3, 18, 60.0, 4, 6, False, 1),   # intervals in slices
    (15000, 1, 2, 512, 2, 4, 190.0, 4, 0, False, 64),   # frames read through L1, rows in slices
    (15000, 1, 2, 64, 2, 3, 20.0, 8, 0, True, 64),      # mixed from there
    (3000, 2, 2, 64, 2, 5, 20.0, 4, 0, False, 64),      # frames as bytes in shared memory
    (3001, 1, 1, 128, 2, 5, 20.0, 8, 0, False, 64),
    (3000, 1, 2, 64, 2, 3, 20.0, 4, 0, True, 64),       # mixed samples in more than a third of an SM
    (70000, 1, 1, 32, 2, 3, 8.0, 8, 0, False, 64),      # frames read through L1
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_box_rows_and_columns(case):
    A, C, P, N, K, T, diam, bits, sub, mix, mb = case
    cfg = synth.small_config(n_ant=A, n_chan=C, n_pol=P, grid_n=N, gcf_k=K, n_time=T, seed=A + T, diameter_m=diam,
                             sigma=0.7)
    cfg = dataclasses.replace(cfg, input_bits=bits, sub_int=sub)
    if mix:
        cfg = dataclasses.replace(cfg, jones=synth.make_jones(cfg, seed=3, gain_rms=0.2, leak_rms=0.2))
    v = synth.random_bytes((T, C, A, P) + ((2,) if bits == 8 else ()), seed=A)
    ref = oracle_image(cfg, v)
    with E.Plan.from_config(cfg, path="plain", max_time=T) as plan:
        d = torch.from_numpy(v).cuda()
        got = plan.image(d)
        a = got.cpu().numpy()
        for mbs in (mb, 512):                    # several chunks, one chunk
            plan.set_param("chunk_mb", mbs)
            b = plan.image(d).cpu().numpy()
            assert np.linalg.norm(b - a) <= 1e-6 * np.linalg.norm(a)
        twice = plan.image(d, out=got, accumulate=True).cpu().numpy()
        plan.sync()
    assert np.allclose(twice, 2 * a, rtol=1e-6, atol=1e-6 * np.abs(a).max())
    for k, (g, r) in enumerate(zip(a, ref) if sub else [(a, ref)]):
        assert_parity(g, r, "plain", f"{case} set {k}")


@pytest.mark.parametrize("case", [
    # A, C, P, N, K, T, diameter, bits: one frame a block where two would leave the chip empty, both forms of the gather
    (300, 41, 2, 32, 4, 3, 7.0, 4), (300, 41, 1, 32, 4, 3, 7.0, 8), (9000, 3, 2, 32, 2, 1, 7.0, 4),
    (400, 4, 2, 64, 7, 1, 24.0, 4),     # two all the same: a batch of one frame has twice the rows
], ids=lambda c: "-".join(str(x) for x in c))
def test_short_launches(case):
    A, C, P, N, K, T, diam, bits = case
    cfg = synth.small_config(n_ant=A, n_chan=C, n_pol=P, grid_n=N, gcf_k=K, n_time=T, seed=A + T, diameter_m=diam, sigma=0.7)
    cfg = dataclasses.replace(cfg, input_bits=bits)
    v = synth.random_bytes((T, C, A, P) + ((2,) if bits == 8 else ()), seed=A)
    with E.Plan.from_config(cfg, path="plain", max_time=T) as plan:
        got = plan.image(torch.from_numpy(v).cuda()).cpu().numpy()
        plan.sync()
    assert_parity(got, oracle_image(cfg, v), "plain", str(case))


@pytest.mark.parametrize("case", [
    # A, C, P, N, K, T, diameter, sub, chunk: intervals cut into slices
    (20, 3, 2, 8, 2, 8, 3.0, 8, 64), (20, 2, 1, 32, 3, 66, 7.0, 33, 64), (30, 1, 2, 64, 3, 300, 17.0, 100, 1),
    (25, 1, 2, 256, 3, 26, 60.0, 13, 64), (25, 1, 1, 512, 2, 18, 120.0, 9, 16),
], ids=lambda c: "-".join(str(x) for x in c))
def test_cut_intervals(case):
    A, C, P, N, K, T, diam, sub, mb = case
    cfg = synth.small_config(n_ant=A, n_chan=C, n_pol=P, grid_n=N, gcf_k=K, n_time=T, seed=A + T, diameter_m=diam, sigma=0.7)
    cfg = dataclasses.replace(cfg, sub_int=sub)
    v = synth.random_bytes((T, C, A, P), seed=A)
    ref = oracle_image(cfg, v)
    with E.Plan.from_config(cfg, path="plain", max_time=T) as plan:
        d = torch.from_numpy(v).cuda()
        assert plan.info()["n_kernels"] == 3
        got = plan.image(d)
        a = got.cpu().numpy()
        plan.set_param("chunk_mb", mb)
        b = plan.image(d).cpu().numpy()
        assert np.linalg.norm(b - a) <= 1e-6 * np.linalg.norm(a)
        plan.image(d, out=got)
        twice = plan.image(d, out=got, accumulate=True).cpu().numpy()
        plan.sync()
    assert np.allclose(twice, 2 * b, rtol=1e-6, atol=1e-6 * np.abs(a).max())
    for k, (g, r) in enumerate(zip(a, ref)):
        assert_parity(g, r, "plain", f"{case} set {k}")


@pytest.mark.parametrize("case", [
    # A, C, P, N, K, T, diameter, bits: more elements than the staged form takes in long launches, staged in these
    (1900, 30, 2, 32, 3, 5, 7.0, 4), (2000, 2, 2, 64, 7, 5, 24.0, 8), (1900, 60, 2, 32, 3, 16, 7.0, 4),
], ids=lambda c: "-".join(str(x) for x in c))
def test_short_launches_of_many_elements(case):
    test_short_launches(case)
