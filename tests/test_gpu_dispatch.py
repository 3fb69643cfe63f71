"""Edges of the size rules by which the library picks a kernel variant or the shape of a launch, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2605_11354_b200 import workloads as wk

import parity_util as pu
from test_gpu_parity import oracle_subset, small_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block,batch,heads,tokens", [(64, 37, 12, 128), (64, 89, 5, 65), (64, 23, 29, 200), (128, 89, 5, 100)])
def test_attention_grids_around_the_number_of_resident_ctas(block, batch, heads, tokens):
    """444, 445, 1334 and 445 attention tiles: three per SM are resident, from one more on CTAs take over tiles."""
    wl = small_workload(f"steal{batch}", batch=batch, heads=heads, tokens=tokens, block=block, crit=0.5, neg=0.3)
    inputs = wk.make_inputs(wl)
    eng, out = pu.run_gpu(inputs, wl)
    ref = oracle_subset(inputs, wl, list(range(heads)), cls=eng.plan.cls.cpu().numpy())
    rel, mx = pu.output_errors(out.cpu().numpy(), ref["out"])
    assert rel <= pu.REL_L2_TOL and mx <= pu.MAX_ABS_TOL
    again = torch.empty_like(out)
    eng.forward(torch.from_numpy(inputs["proj"]).cuda(), out=again)
    assert torch.equal(again, out)  # whichever CTA computes a tile


@pytest.mark.parametrize("block", [64, 128])
def test_many_buffer_sets_in_turn(block):
    """Encoded tensor maps are kept for a few hundred buffers: more sets than that, at addresses that come and go, give the
    same bytes."""
    wl = small_workload(f"maps{block}", heads=2, tokens=300, block=block)
    inputs = wk.make_inputs(wl)
    first, hold = None, []
    for i in range(400):
        eng, out = pu.run_gpu(inputs, wl)
        first = out.clone() if first is None else first
        assert torch.equal(out, first)
        if i % 3:
            hold.append(eng)  # some buffers stay, the others' addresses are taken over
