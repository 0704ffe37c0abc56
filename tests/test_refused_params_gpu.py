"""A refused tuning parameter leaves the plan as it was: the same parameters and bit-equal images."""
import pytest

import epic_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402

GRID = ("grid_kernel", "grid_frames")


def test_refused_gridding_kernel_leaves_the_tensor_core_one_as_it_was():
    # the tallest SKA-Low channel: the balanced kernel's tiles, tasks and entries do not fit, and trying
    # them configures the pair-list kernel on the way
    cfg = synth.config(3).subset([383], n_time=20)
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan.from_config(cfg, path="dftgemm") as plan:
        before = {k: plan.get_param(k) for k in GRID}
        assert before["grid_kernel"] == 4
        for bad in (2, 0, 5):
            with pytest.raises(E.EpicError) as ex:
                plan.set_param("grid_kernel", bad)
            assert ex.value.status == 7
            assert {k: plan.get_param(k) for k in GRID} == before, bad
        got = plan.image(v)       # a launch out of step with its configuration is an error, not a kernel
        plan.sync()
        with E.Plan.from_config(cfg, path="dftgemm") as fresh:
            assert torch.equal(got, fresh.image(v))
            fresh.sync()
        plan.set_param("grid_kernel", 3)
        plan.set_param("grid_kernel", 4)
        assert plan.get_param("grid_kernel") == 4
        assert torch.equal(got, plan.image(v))
        plan.sync()


def test_refused_frames_of_the_pair_list_kernel_leave_its_staging_as_it_was():
    # 2430 dual-pol elements: the lists fit beside four frames of voltages, eight frames do not fit at all
    cfg = synth.small_config(n_ant=2430, n_chan=2, n_pol=2, grid_n=128, gcf_k=2, n_time=5, seed=8, diameter_m=60.0,
                             sigma=0.7)
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan.from_config(cfg, path="dftgemm", max_time=5) as plan:
        plan.set_param("grid_kernel", 3)
        plan.set_param("grid_frames", 4)
        before = plan.image(v)
        with pytest.raises(E.EpicError) as ex:
            plan.set_param("grid_frames", 8)
        assert ex.value.status == 7
        assert plan.get_param("grid_frames") == 4
        assert torch.equal(plan.image(v), before)
        plan.sync()


def test_scratch_that_cannot_be_had_leaves_the_plan_working():
    # 100,000 samples of 64 channels as tiles are more than the device's memory
    cfg = synth.small_config(n_ant=40, n_chan=64, n_pol=2, grid_n=128, gcf_k=3, n_time=20, seed=31, diameter_m=85.0)
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan.from_config(cfg, path="dftgemm", max_time=100_000) as plan:
        before = plan.image(v)
        info, budget = plan.info(), plan.get_param("chunk_mb")
        with pytest.raises(E.EpicError) as ex:
            plan.set_param("chunk_mb", 2_000_000)
        assert ex.value.status == 3               # EPIC_ERR_OOM
        assert plan.info() == info and plan.get_param("chunk_mb") == budget
        for _ in range(2):                        # no error left over for the next calls
            assert torch.equal(plan.image(v), before)
            plan.sync()


def test_frames_that_the_gather_kernels_take_stay_valid():
    # 600 dual-pol elements: the tensor-core kernel stages two groups at most
    cfg = synth.small_config(n_ant=600, n_chan=2, n_pol=2, grid_n=64, gcf_k=3, n_time=70, seed=9, diameter_m=25.0)
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan.from_config(cfg, path="dftgemm") as plan:
        assert plan.get_param("grid_kernel") == 4 and plan.get_param("grid_frames") == 2
        want = plan.image(v)
        for F in (4, 8, 1):
            plan.set_param("grid_frames", F)
            assert plan.get_param("grid_frames") == F
            assert torch.equal(plan.image(v), want)
            plan.sync()
