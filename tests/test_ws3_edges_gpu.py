"""k_dftgemm_ws3 at the edges of its tiles and of its cuts of the work."""
import dataclasses

import numpy as np
import pytest

import epic_synth as synth
from gpu_common import assert_parity, oracle_image

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


def make(A, C, P, N, T, diam, sub=0, max_time=None):
    cfg = synth.small_config(n_ant=A, n_chan=C, n_pol=P, grid_n=N, gcf_k=4, n_time=T, seed=A + T, diameter_m=diam,
                             sigma=0.7)
    cfg = dataclasses.replace(cfg, sub_int=sub)
    plan = E.Plan(cfg.pos_m, cfg.freq_hz, P, N, 4, cfg.sigma_cells, cfg.f_ref_hz, False, None, "dftgemm",
                  max_time or max(T, 16), sub_int=sub)
    return cfg, plan, synth.random_bytes((T, C, A, P), seed=A)


# boxes from one 8-cell chunk a row to many: every width of the panels that end an unpadded row
@pytest.mark.parametrize("P", [1, 2])
@pytest.mark.parametrize("diam", [2.0, 9.0, 17.0, 26.0, 34.0, 43.0, 51.0, 60.0, 68.0, 77.0, 85.0])
def test_unpadded_tiles(diam, P):
    cfg, plan, vn = make(30, 2, P, 128, 20, diam)
    with plan:
        v = torch.from_numpy(vn).cuda()
        assert plan.get_param("grid_kernel") == 4
        got = plan.image(v).cpu().numpy()
        plan.set_param("grid_kernel", 1)          # padded tiles
        ref = plan.image(v).cpu().numpy()
        plan.sync()
    assert_parity(got, oracle_image(cfg, vn), "dftgemm", str(plan.n_pol))
    # the grid sums differ by FP32 rounding, so that about 1e-4 of the FP16 tile values round the other way
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)


SPLITS = [
    # A, C, P, N, T, diameter
    (12, 1, 2, 64, 900, 12.0),    # one item on every block: parts added in two levels
    (12, 1, 1, 64, 331, 12.0),
    (20, 2, 2, 128, 60, 20.0),    # a run of fewer blocks than the others
    (40, 3, 2, 256, 21, 40.0),    # eight blocks side by side
    (40, 2, 2, 128, 7, 85.0),     # row parts, fewer frames than blocks
    (16, 3, 2, 32, 1, 8.0),       # one frame
    (16, 5, 1, 8, 3, 3.0),        # an image smaller than a warp's rows
]


@pytest.mark.parametrize("case", SPLITS, ids=lambda c: "-".join(str(x) for x in c))
def test_cuts_agree(case):
    A, C, P, N, T, diam = case
    cfg, plan, vn = make(*case)
    with plan:
        v = torch.from_numpy(vn).cuda()
        got = {}
        for split in (-1, 0, 1):
            plan.set_param("split", split)
            got[split] = plan.image(v).cpu().numpy()
            again = torch.zeros(plan.image_shape(T), device="cuda")
            for _ in range(2):                    # the counters are ready for the next launch
                plan.image(v, out=again, accumulate=True)
            plan.sync()
            assert np.array_equal(again.cpu().numpy(), 2 * got[split])
    # the same frames' products in FP32 sums of another order
    tol = max(T, 8) * 2.0 ** -24
    for split in (-1, 1):
        assert np.linalg.norm(got[split] - got[0]) <= tol * np.linalg.norm(got[0]), split


@pytest.mark.parametrize("case", [(12, 5, 2, 128, 24, 20.0, 3), (12, 1, 2, 64, 320, 12.0, 2), (12, 3, 1, 32, 18, 8.0, 18),
                                  (40, 2, 2, 256, 10, 85.0, 1), (16, 4, 2, 8, 12, 3.0, 4)],
                         ids=lambda c: "-".join(str(x) for x in c))
def test_sub_integrations_cut_between_intervals(case):
    A, C, P, N, T, diam, sub = case
    cfg, plan, vn = make(*case)
    v = torch.from_numpy(vn).cuda()
    with plan:
        got = plan.image(v).cpu().numpy()
        twice = torch.from_numpy(got).cuda()
        plan.image(v, out=twice, accumulate=True)
        plan.sync()
    assert np.array_equal(twice.cpu().numpy(), 2 * got)
    _, whole, _ = make(A, C, P, N, T, diam)
    with whole:
        for i in range(T // sub):
            one = whole.image(v[i * sub:(i + 1) * sub].contiguous()).cpu().numpy()
            whole.sync()
            tol = max(sub, 8) * 2.0 ** -24
            assert np.linalg.norm(got[i] - one) <= tol * np.linalg.norm(one), i
