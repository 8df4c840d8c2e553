"""Tiles whose items each compute a share of the output's columns (fewer tiles than the device has SM pairs), against the oracle: four
items or two to a chunk, one chunk and two, last tiles without their second half; and the merge kernel with four rows of a warp one
after the other, which takes more than 74 tiles of several chunks."""
import pytest

from paper_2609_24698_b200 import synth
from tests.test_gpu_parity import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,topk,lengths", [
    (1, 5, 600, [400]),                                       # two tiles of one chunk: four items each
    (1, 8, 600, [1400]),                                      # of two chunks: eight items, the last merges
    (1, 1, 600, [3]),                                         # a quarter of a tile, hardly a key
    (14, 6, 600, [90 + 100 * i for i in range(14)]),          # 28 tiles: one chunk by two items, two by one each
    (3, 4, 300, [90, 800, 2600]),                             # three tiles, long lists possible: whole, or cut into chunks of 256 keys
    (76, 2, 300, [100 + 25 * i for i in range(76)]),          # 76 tiles of one to three chunks
])
def test_shares_of_columns(B, D, topk, lengths):
    cfg = synth.Config(f"few_{B}_{D}", 217, synth.Shape("bf16", B, D, 64, 512, 2, topk, 2, 128, 16, 128), L_min=1, L_max=max(lengths), layers=1, seed=31 + B)
    lockstep(cfg, cycles=2, lengths=lengths, want_topk=False)
