"""The stored tiles of the batched mix lose to no default: a batch whose plans took
them runs no longer than the same batch on the library's own choice (5 % is left
for the timing)."""
import pytest

from paper_1811_04165_gb300 import synth

pytestmark = pytest.mark.gpu


def test_stored_tiles_do_not_lose_to_the_default(lib):
    import torch
    from paper_1811_04165_gb300 import batch_study
    wls = synth.batch_beams(4, seed=5, dm_trials=(512, 1024), max_widths=4)
    times = []
    for tuned in (False, True):
        plans = [lib.Plan.from_workload(w) for w in wls]
        if tuned:
            assert batch_study.apply_tuned(plans) == len(plans)
        xs = [torch.randint(0, 256, (p.channels, p.pitch), dtype=torch.uint8, device="cuda") for p in plans]
        batch = lib.Batch(plans, xs, branches=4)
        times.append(min(batch_study._time(batch.launch, 10) for _ in range(3)))
        del batch
    assert times[1] <= 1.05 * times[0], times
