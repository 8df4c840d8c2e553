"""Merging of tiles of several chunks, with the tiles few (cut to fill the device, merged when all are done) and many (each merged as
soon as its chunks are stored), against the oracle: one to five chunks side by side, a last tile without its second half."""
import pytest

from paper_2609_24698_b200 import synth
from tests.test_gpu_parity import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,lengths", [(2, 3, [3700, 900]), (19, 6, [100 + 190 * i for i in range(19)]), (40, 2, [60 + 97 * i for i in range(40)])])
def test_merge_of_few_and_many_tiles(B, D, lengths):
    cfg = synth.Config(f"merge_{B}_{D}", 213, synth.Shape("bf16", B, D, 64, 512, 2, 600, 2, 128, 16, 128), L_min=50, L_max=max(lengths), layers=2, seed=11 + B)
    lockstep(cfg, cycles=2, lengths=lengths, want_topk=False)
