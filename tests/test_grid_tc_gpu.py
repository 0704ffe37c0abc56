"""Tensor-core gridding (grid_kernel 4) against the FP32 gather kernel and the oracle."""
import dataclasses

import numpy as np
import pytest

import epic_synth as synth
from gpu_common import assert_parity, oracle_image

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402

CASES = [
    # A, C, P, N, K, T, diameter, bits, table oversampling, mixing
    (40, 3, 2, 64, 3, 37, 18.0, 4, 0, False),     # a ragged second group of frames
    (25, 2, 1, 32, 3, 70, 9.0, 4, 0, False),      # one pol: groups of 64 frames; odd frame bytes
    (33, 3, 2, 64, 4, 65, 18.0, 8, 0, False),
    (21, 2, 1, 64, 5, 130, 20.0, 8, 0, False),
    (80, 3, 2, 128, 5, 40, 85.0, 4, 0, False),    # row parts with padding rows
    (250, 2, 2, 64, 7, 100, 12.0, 4, 0, False),   # dense: tiles of more K steps than the ring holds
    (6, 2, 2, 8, 3, 20, 3.0, 4, 0, False),        # fewer frames than a group, one tile
    (30, 2, 2, 64, 4, 33, 18.0, 4, 8, False),     # complex weights
    (29, 2, 1, 64, 3, 129, 18.0, 4, 4, False),
    (31, 2, 1, 64, 3, 50, 18.0, 8, 4, False),
    (40, 3, 2, 64, 3, 37, 18.0, 4, 0, True),      # mixed voltages split into hi and lo
    (33, 3, 2, 64, 4, 65, 18.0, 8, 0, True),
    (30, 2, 2, 64, 4, 33, 18.0, 4, 8, True),
]


def make(case):
    A, C, P, N, K, T, diam, bits, tab, mix = case
    cfg = synth.small_config(n_ant=A, n_chan=C, n_pol=P, grid_n=N, gcf_k=K, n_time=T, seed=A + T, diameter_m=diam,
                             sigma=0.7)
    cfg = dataclasses.replace(cfg, input_bits=bits)
    if mix:
        cfg = dataclasses.replace(cfg, jones=synth.make_jones(cfg, seed=3, gain_rms=0.2, leak_rms=0.2))
    kw = {}
    if tab:
        d = np.arange(K * tab + 1) / tab - 0.5 * K
        x, y = np.meshgrid(d, d)
        w = (np.exp(-(x * x + y * y) / 1.2) * np.exp(1j * (0.3 * x - 0.2 * y))).astype(np.complex64)
        kw = {"gcf_table": w.view(np.float32), "oversample": tab}
    plan = E.Plan(cfg.pos_m, cfg.freq_hz, P, N, K, cfg.sigma_cells, cfg.f_ref_hz, False, None, "dftgemm", T,
                  input_bits=bits, jones=cfg.jones, **kw)
    v = synth.random_bytes((T, C, A, P) + ((2,) if bits == 8 else ()), seed=A)
    return cfg, plan, v, tab


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_tensor_core_gridding(case):
    cfg, plan, vn, tab = make(case)
    with plan:
        assert plan.get_param("grid_kernel") == 4
        v = torch.from_numpy(vn).cuda()
        got = plan.image(v).cpu().numpy()
        plan.sync()
        for F in (1, 2, 4):                      # groups staged at once: the same sums
            try:
                plan.set_param("grid_frames", F)
            except E.EpicError as ex:
                assert ex.status == 7
                continue
            assert np.array_equal(plan.image(v).cpu().numpy(), got), F
        raw = torch.zeros(v.numel() + 16, dtype=torch.uint8, device="cuda")
        for off in (1, 2):                       # frames that start at any byte
            va = raw[off:off + v.numel()].view(v.shape)
            va.copy_(v)
            assert np.array_equal(plan.image(va).cpu().numpy(), got), off
        short = plan.image(v[:5].contiguous()).cpu().numpy()   # a block far shorter than a group
        plan.set_param("grid_kernel", 1)
        ref = plan.image(v).cpu().numpy()
        ref5 = plan.image(v[:5].contiguous()).cpu().numpy()
        plan.sync()
    # grid sums differ by FP32 rounding, so about 1e-4 of the FP16 tile values round the other way
    # (2^-11 each), which the two transforms spread to 2e-5 of a frame's images: less in a sum of frames
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
    assert np.linalg.norm(short - ref5) <= 2e-5 * np.linalg.norm(ref5)
    if not tab:
        assert_parity(got, oracle_image(cfg, vn), "dftgemm", str(case))
