"""Images at any float of an allocation: the same values as in a buffer that begins at 16 bytes."""
import pytest

import epic_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


def check(plan, v):
    want = plan.image(v)
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
