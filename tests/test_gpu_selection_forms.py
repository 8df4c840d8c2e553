"""The two forms of the selection over lists beyond the short ones (one cluster per sequence; scores over all SMs and a CTA per
node), at the edges of their ranges, against the oracle."""
import pytest

from paper_2609_24698_b200 import synth
from tests.test_gpu_parity import _plant_tied_indexer_keys, lockstep

pytestmark = pytest.mark.gpu


# entries = L / 2: one past the short lists; shares of the eight CTAs that are whole sixteens, one more, one less; the longest list
# of the cluster form and the first of the other; more than eight nodes (the other form at any length); a tiny last share
@pytest.mark.parametrize("D,HI,lengths", [(8, 4, [1560, 2047, 2048, 2050]), (5, 1, [1537, 4096, 4130, 260]), (8, 2, [8150, 8145, 700, 5000]),
                                          (8, 3, [8192, 8204, 16500, 90]), (12, 4, [1600, 3001, 4500, 300]), (17, 2, [2048, 2563, 4400, 64])])
@pytest.mark.parametrize("ties", [False, True])
def test_selection_forms_at_the_edges(D, HI, lengths, ties):
    cfg = synth.small_config(name=f"sel_forms_{D}_{HI}_{max(lengths)}", dtype="bf16", B=4, D=D, H=4, d=16, m_csa=2, topk=130, HI=HI, di=128,
                             m_hca=32, window=32, L_min=64, L_max=max(lengths), layers=1, seed=31 + D + HI, cfg_id=210)
    lockstep(cfg, cycles=1, lengths=lengths, plant=_plant_tied_indexer_keys(every=40) if ties else None, exact_topk=ties)


@pytest.mark.parametrize("page_tokens", [0, 64])
def test_selection_forms_without_index_lists(page_tokens):
    """The tensor-core path reads mask rows only: both forms without a buffer for the index lists, flat and paged."""
    for topk, L in ((64, [900, 3300, 40, 2900]), (300, [33200, 1500])):
        cfg = synth.Config(f"sel_forms_masks_{topk}", 211, synth.Shape("bf16", len(L), 8, 64, 512, 4 if topk == 300 else 2, topk, 4, 128, 64, 128),
                           L_min=40, L_max=max(L), seed=7)
        lockstep(cfg, cycles=1, lengths=L, want_topk=False, page_tokens=page_tokens)
