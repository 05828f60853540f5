"""The wide tile of the pre-summed pass folds its lanes at most 17 times (its 8-bit
counts take 15 per fold), checked by the library's verifier on the chunk lists it
builds (no GPU): bands of many channels at delays so short that chunks hold all
units that a chunk may, and longer ones, where windows decide."""
import pytest

import oracle
from paper_1811_04165_gb300 import synth


@pytest.mark.parametrize("C", [3240, 3244, 3600, 4093, 4096])
@pytest.mark.parametrize("step", [0.001, 0.002, 0.02])
def test_folds(lib, C, step):
    d = oracle.delay_table(1250.0, 1550.0, C, 81.92e-6, synth.dm_grid(130, step))
    lib.sps_presum_tables_verify(d, C, 12560, lib.DedispConfig(4, 16, 8, 1, 16, 2))


@pytest.mark.parametrize("chunk,presum", [(64, 1), (48, 1), (32, 1), (64, 2), (10, 1)])
def test_chunks_hold_what_their_stage_is_sized_for(lib, chunk, presum):
    d = oracle.delay_table(1250.0, 1550.0, 389, 81.92e-6, synth.dm_grid(70, 0.05))
    lib.sps_presum_tables_verify(d, 389, 2000, lib.DedispConfig(4, 8, 4, 1, chunk, presum))
