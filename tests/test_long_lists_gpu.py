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
