"""Captured kicks in each gather order that the autotuner may choose, forces by
sorted slot (gather_rows = 2) among them: the graph's velocities are those of the
direct launches, bit for bit, and of the other orders."""
import numpy as np
import pytest

from paper_1209_0461_gb300 import batch, synth

pytestmark = pytest.mark.gpu


def test_captured_kicks_in_every_gather_order():
    import torch
    boxes = synth.batched_boxes(3, n_hist=8, n_kbins=32)
    runs = []
    for rows in (0, 1, 2):
        b = batch.Batch(boxes, n_streams=2, autotune=False)
        for it in b.items:
            it["pm"].set_tuning(gather_rows=rows)
        for step in (b.eager_step, None):
            if step is None:
                b.capture()
                b.reset_velocities()
                step = b.step
            step()
            b.check()
            torch.cuda.synchronize()
            runs.append([(it["vel"] - it["vel0"]).cpu().numpy() for it in b.items])
            b.reset_velocities()
        b.close()
    for other in runs[1:]:
        for d0, d1 in zip(runs[0], other):
            assert np.any(d0 != 0) and np.array_equal(d0, d1)
