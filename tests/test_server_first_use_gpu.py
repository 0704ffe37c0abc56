"""A server's first blocks: slots take their call memory while other slots' kernels run."""
import dataclasses

import numpy as np
import pytest

import epic_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_03027_gb300 as E  # noqa: E402


def test_first_blocks_of_fresh_slots_equal_the_plan_alone():
    # every slot's memory is allocated and zeroed with its first block; the zeros must not land on
    # tiles, or on the counters of split work items, that the block's kernels already wrote
    types = synth.mixed_station_types()[1:3]
    plans, blocks, alone = [], [], []
    for k, st in enumerate(types):
        cfg = dataclasses.replace(synth.serving_config(st, 64), n_time=96)
        v = torch.from_numpy(synth.random_bytes((96, 64, cfg.n_ant, cfg.n_pol), seed=70 + k)).pin_memory()
        plan = E.Plan.from_config(cfg, path="dftgemm", max_time=96)
        alone.append(plan.image(v.cuda()).cpu().numpy())
        plan.sync()
        plans.append(plan)
        blocks.append(v)
    for _ in range(3):
        with E.Server(1 << 30, 4) as srv:
            outs = [torch.empty(plans[i % 2].image_shape(96), device="cuda") for i in range(8)]
            torch.cuda.synchronize()
            tickets = [srv.submit_ptr(plans[i % 2], blocks[i % 2].data_ptr(), 96, outs[i]) for i in range(8)]
            for t in tickets:
                srv.wait(t)
            for i, o in enumerate(outs):
                assert np.array_equal(o.cpu().numpy(), alone[i % 2]), i
    for p in plans:
        p.close()
