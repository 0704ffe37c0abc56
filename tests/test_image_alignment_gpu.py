"""Images at any float of an allocation: the same values as in a buffer that begins at 16 bytes."""
import numpy as np
import pytest

import epic_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


def check(plan, v, want=None):
    want = plan.image(v) if want is None else want
    n = want.numel()
    raw = torch.full((n + 8,), 5.0, device="cuda")
    for off in (1, 2, 3):
        out = raw[off:off + n].view(want.shape)
        assert out.data_ptr() % 16 == 4 * off
        plan.image(v, out=out)
        assert torch.equal(out, want), off
        plan.image(v, out=out, accumulate=True)
        assert torch.equal(out, 2 * want), off
        plan.sync()
        assert (raw[:off] == 5.0).all() and (raw[off + n:] == 5.0).all()
        raw.fill_(5.0)


@pytest.mark.parametrize("P,N,T", [(2, 64, 67), (1, 128, 45), (2, 8, 40)])
def test_plain_path_with_slices_of_the_frames(P, N, T):
    cfg = synth.small_config(n_ant=30, n_chan=1, n_pol=P, grid_n=N, gcf_k=3, n_time=T, seed=N, diameter_m=0.25 * N,
                             sigma=0.7)
    with E.Plan.from_config(cfg, path="plain") as plan:
        assert plan.info()["n_kernels"] == 3      # rows, columns and the sum of the slices
        check(plan, torch.from_numpy(synth.make_voltages(cfg)).cuda())


@pytest.mark.parametrize("P,N,T,sub", [(2, 8, 20, 0), (1, 16, 20, 0), (2, 64, 40, 0), (2, 128, 12, 3), (1, 256, 5, 0), (2, 8, 8, 2)])
def test_tensor_path(P, N, T, sub):
    # such images take whole items (intervals) of the default kernel whatever kernel and cut the plan has
    cfg = synth.small_config(n_ant=24, n_chan=2, n_pol=P, grid_n=N, gcf_k=3, n_time=T, seed=N + T, diameter_m=0.2 * N,
                             sigma=0.7)
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan(cfg.pos_m, cfg.freq_hz, P, N, 3, cfg.sigma_cells, cfg.f_ref_hz, False, None, "dftgemm", T,
                sub_int=sub) as plan:
        if not sub:
            plan.set_param("split", 0)
        want = plan.image(v)
        check(plan, v, want)
        for name, value in ([] if sub else [("split", 1), ("mma_kernel", 1), ("mma_kernel", 2)]):
            plan.set_param(name, value)
            check(plan, v, want)


def test_tensor_path_of_the_slab_kernel():
    # a box too wide for the warp-specialised kernels
    cfg = synth.small_config(n_ant=24, n_chan=1, n_pol=1, grid_n=512, gcf_k=2, n_time=4, seed=3, sigma=0.7)
    cell = 0.5 * 299792458.0 / cfg.freq_hz[0]
    pos = np.stack([np.linspace(-168.0, 168.0, 24), 3.0 * np.sin(np.arange(24.0))], axis=1) * cell
    v = torch.from_numpy(synth.make_voltages(cfg)).cuda()
    with E.Plan(pos, cfg.freq_hz, 1, 512, 2, cfg.sigma_cells, cfg.f_ref_hz, False, None, "dftgemm", 4) as plan:
        assert plan.info()["tc_kernel"] == 5
        check(plan, v)
