"""fp32 storage with 128-wide rows: the cluster attention kernel and the fp32 form of the cluster selection, at the edges of their
splits, against the oracle."""
import pytest

from paper_2609_24698_b200 import synth
from tests.test_gpu_parity import _plant_tied_indexer_keys, lockstep

pytestmark = pytest.mark.gpu


# B, D, H, HI, topk, m_csa, window, lengths: eight CTAs a node with shares of a few keys; heads that do not fill a group; shares of one
# tile, one key more, many tiles (one CTA a node); more nodes than the cluster selection takes; no key but the node itself
@pytest.mark.parametrize("B,D,H,HI,topk,m_csa,window,lengths,page", [
    (1, 5, 16, 1, 64, 4, 128, [1024], 0), (2, 8, 20, 2, 30, 2, 16, [0, 333], 0), (3, 6, 5, 4, 100, 2, 32, [260, 1201, 77], 32),
    (16, 8, 33, 1, 64, 4, 128, [130 + 251 * i for i in range(16)], 0), (40, 8, 16, 3, 200, 2, 64, [400 + 13 * i for i in range(40)], 0),
    (2, 12, 16, 2, 40, 2, 16, [640, 1500], 0), (1, 8, 16, 1, 900, 2, 128, [8100], 0)])
def test_f32_attention_and_selection(B, D, H, HI, topk, m_csa, window, lengths, page):
    cfg = synth.Config(f"f32_{B}_{D}_{H}", 213, synth.Shape("fp32", B, D, H, 128, m_csa, topk, HI, 64, 32, window), L_min=0, L_max=max(lengths), seed=B + H)
    lockstep(cfg, cycles=2, lengths=lengths, page_tokens=page)


def test_f32_selection_exact_ties():
    """(Keys of 8 bits, so that the oracle's own fp64 sums are exact whatever order its matrix product takes.)"""
    tie = _plant_tied_indexer_keys(every=40)

    def plant(states, lengths):
        tie(states, lengths)
        for S in (S for layer in states for S in layer):
            S.csa_ik[:] = synth.quantize(S.csa_ik, "bf16")
    cfg = synth.Config("f32_ties", 214, synth.Shape("fp32", 3, 6, 4, 128, 2, 100, 2, 64, 32, 16), L_min=0, L_max=4000, seed=3)
    lockstep(cfg, cycles=1, lengths=[700, 2600, 4000], plant=plant, exact_topk=True)


@pytest.mark.parametrize("scale", [3.0, 40.0])
def test_f32_peaked_softmax_over_many_tiles(scale):
    cfg = synth.Config("f32_peaked", 215, synth.Shape("fp32", 8, 8, 64, 128, 2, 500, 1, 64, 32, 128, scale), L_min=0, L_max=3000, seed=5)
    lockstep(cfg, cycles=1, lengths=[3000, 2501, 64, 130, 900, 1027, 2048, 333])


# Selections that outweigh the keys known before them: two CTAs an SM, in clusters of eight, four (the most that there are), two; one
# where there are more nodes than places; capacities in which no node ranks, whose keys are one list, in shares of a few keys and of many
@pytest.mark.parametrize("B,D,topk,lengths", [
    (4, 8, 500, [1300, 1041, 90, 0]), (8, 8, 400, [900 + 31 * i for i in range(8)]), (9, 8, 400, [1000 - 7 * i for i in range(9)]),
    (18, 8, 256, [600 + 20 * i for i in range(18)]), (40, 8, 300, [700 + 9 * i for i in range(40)]), (1, 5, 1000, [700]), (16, 7, 1000, [64 * i + i for i in range(16)]),
    (40, 8, 600, [25 * i for i in range(40)])])
def test_f32_selections_that_outweigh_the_rest(B, D, topk, lengths):
    cfg = synth.Config(f"f32_chosen_{B}_{topk}", 218, synth.Shape("fp32", B, D, 16, 128, 2, topk, 1, 64, 32, 32), L_min=0, L_max=max(lengths), seed=B + topk)
    lockstep(cfg, cycles=2, lengths=lengths)
