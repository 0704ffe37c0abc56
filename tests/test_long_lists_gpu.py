"""Gridding with lists too long for the balanced kernel's tasks: the pair lists hold every channel all the same."""
import numpy as np
import pytest

import epic_synth as synth
from gpu_common import assert_parity, oracle_image

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


@pytest.mark.parametrize("T", [4, 20])
def test_pair_lists_of_every_channel_where_task_lists_are_too_long(T):
    # 700 elements over 12 x 12 cells of a 32 x 32 grid: more than 255 of them reach a cell pair
    cfg = synth.small_config(n_ant=700, n_chan=6, n_pol=2, grid_n=32, gcf_k=5, n_time=T, seed=12, diameter_m=8.0,
                             sigma=0.7)
    vn = synth.make_voltages(cfg)
    ref = oracle_image(cfg, vn)
    v = torch.from_numpy(vn).cuda()
    with E.Plan.from_config(cfg, path="dftgemm") as plan:
        with pytest.raises(E.EpicError) as ex:
            plan.set_param("grid_kernel", 2)
        assert ex.value.status == 7
        plan.set_param("grid_kernel", 3)
        got = plan.image(v).cpu().numpy()
        plan.sync()
    assert np.all(np.isfinite(got))
    assert_parity(got, ref, "dftgemm", f"T={T}")


@pytest.mark.parametrize("tab", [0, 4])
@pytest.mark.parametrize("T", list(range(1, 12)))
def test_short_passes_of_the_row_major_kernel(T, tab):
    # a pass of fewer frames than the kernel's goes by powers of two of them: the same sums in the same order
    cfg = synth.small_config(n_ant=70, n_chan=2, n_pol=2, grid_n=32, gcf_k=3, n_time=T, seed=14, diameter_m=8.0, sigma=0.7)
    kw = {}
    if tab:
        d = np.arange(3 * tab + 1) / tab - 1.5
        x, y = np.meshgrid(d, d)
        kw = {"gcf_table": (np.exp(-(x * x + y * y)) * np.exp(1j * (0.3 * x - 0.2 * y))).astype(np.complex64).view(np.float32),
              "oversample": tab}
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan(cfg.pos_m, cfg.freq_hz, 2, 32, 3, cfg.sigma_cells, cfg.f_ref_hz, False, None, "dftgemm", 15, **kw) as plan:
        if not tab:
            plan.set_param("grid_kernel", 1)
        got = []
        for F in (1, 2, 4, 8):
            plan.set_param("grid_frames", F)
            got.append(plan.image(v))
            plan.sync()
        assert all(torch.equal(g, got[0]) for g in got)
        ref = plan.image(v[:1].contiguous())
        for t in range(1, T):
            plan.image(v[t:t + 1].contiguous(), out=ref, accumulate=True)
        plan.sync()
    # the frames' products in FP32 sums of another order
    tol = max(T, 8) * 2.0 ** -24
    assert (got[0] - ref).norm() <= tol * ref.norm()
