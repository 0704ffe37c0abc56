"""Voltages at any byte of an allocation: the same images as from a block that begins at 256 bytes."""
import dataclasses

import pytest

import epic_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("path,P,A,T,kernel", [
    ("plain", 2, 33, 7, 0), ("plain", 1, 21, 6, 0), ("plain", 2, 9000, 2, 0), ("fused", 2, 33, 5, 0), ("fused", 1, 21, 5, 0),
    ("dftgemm", 2, 33, 20, 4), ("dftgemm", 1, 21, 20, 4), ("dftgemm", 2, 33, 5, 1), ("dftgemm", 2, 33, 5, 2), ("dftgemm", 2, 33, 5, 3),
    ("dftgemm", 1, 21, 5, 1), ("dftgemm", 1, 21, 5, 2), ("dftgemm", 1, 21, 5, 3), ("dftgemm", 2, 1800, 5, 0),
])
def test_any_byte(path, P, A, T, kernel, bits):
    cfg = synth.small_config(n_ant=A, n_chan=2, n_pol=P, grid_n=32, gcf_k=3, n_time=T, seed=A + T, diameter_m=9.0, sigma=0.7)
    cfg = dataclasses.replace(cfg, input_bits=bits)
    v = torch.from_numpy(synth.random_bytes((T, 2, A, P) + ((2,) if bits == 8 else ()), seed=A)).cuda()
    raw = torch.zeros(v.numel() + 16, dtype=torch.uint8, device="cuda")
    with E.Plan.from_config(cfg, path=path) as plan:
        if kernel:
            plan.set_param("grid_kernel", kernel)
        want = plan.image(v)
        for off in (1, 2, 3):
            va = raw[off:off + v.numel()].view(v.shape)
            va.copy_(v)
            assert torch.equal(plan.image(va), want), off
            plan.sync()
