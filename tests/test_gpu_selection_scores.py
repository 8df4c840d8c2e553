"""Selections over lists with scores at which a float compare and a total order differ, in every selection form: exactly topk
entries whatever the values, nothing written past a node's row.  The scores are exact small numbers, so that the expected selection
is one sort on the host."""
import numpy as np
import pytest
import torch

from paper_2609_24698_b200 import synth

pytestmark = pytest.mark.gpu

# dtype, nodes, committed entries, topk.  One CTA per node (short lists); a cluster per sequence, bf16 and fp32; scores over all SMs
# and a cluster per node, for more than eight nodes and for a long list; the general kernels (other indexer widths): keys in registers,
# a cluster per node, a list read again in every pass.  The last: so many heads (the sixth number) that nothing is split and the ranges
# of the scores over all SMs have no room among partial outputs
FORMS = [("bf16", 8, 600, 512), ("bf16", 8, 900, 800), ("fp32", 8, 600, 512), ("bf16", 12, 900, 800), ("bf16", 7, 4300, 4200),
         ("fp32", 8, 900, 800, 16), ("bf16", 8, 2500, 2400, 16), ("fp32", 5, 66000, 65800, 8), ("bf16", 20, 900, 800, 128, 256)]


def _select(form, HI, ik, tree_ik, iq, iw, room=None, cap=None, status=0):
    """topk_idx of a chain of D nodes (blocks of two tokens: nodes 1, 3, ... close one) after n committed entries with the indexer
    keys ik [n][di]; every closed entry has the key tree_ik.  The list buffer is followed by a guard.  room: tokens the shape is
    sized for; cap: entries the cache says it has room for; status: what the device has to report."""
    from paper_2609_24698_b200 import harness as hz
    dtype, D, n, k = form[:4]
    di = ik.shape[1]
    sh = synth.Shape(dtype, 1, D, form[5] if len(form) > 5 else 4, 16, 2, k, HI, di, 64, 64)
    ccap, hcap = hz.capacities(sh, [2 * n], 2 * D)
    eng = hz.VerifyEngine(sh, 1, ccap, hcap, room or 2 * n + 2 * D, want_topk=True)
    guard = torch.full((D * k + 64,), -2, dtype=torch.int32, device="cuda")
    eng.topk_idx = [guard[:D * k].view(1, D, k)]
    eng.caches[0].L.fill_(2 * n)
    if cap is not None:
        eng.caches[0].csa_cap.fill_(cap)
    eng.caches[0].csa_ik[:n] = torch.from_numpy(ik).cuda()
    inp = hz.InputSet.empty(sh, 1)
    nd = inp.layers[0]
    nd.parent.copy_(torch.arange(-1, D - 1).view(1, D)); nd.n_nodes.fill_(D)
    nd.ikc[:] = torch.from_numpy(tree_ik).cuda()
    nd.iq[:] = torch.from_numpy(iq).cuda(); nd.iw[:] = torch.from_numpy(iw).cuda()
    eng.launch_cycle(inp, refresh=False)
    torch.cuda.synchronize()
    assert int(eng.status.sum()) == status
    got = guard.cpu().numpy()
    assert (got[D * k:] == -2).all(), "written past the last node's row"
    return got[:D * k].reshape(D, k)


def _check(got, form, scores, tree_score):
    """scores: of the committed entries, tree_score: of every closed one; NaN above everything, ties to the lower index."""
    for node, row in enumerate(got):
        s = np.concatenate([scores, np.full(node // 2, tree_score) if np.isscalar(tree_score) else tree_score])
        order = np.lexsort((np.arange(len(s)), -np.where(np.isnan(s), np.inf, s)))
        assert np.array_equal(row, np.sort(order[:form[3]])), (node, len(set(row.tolist())))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("where", ["committed", "tree"])
@pytest.mark.parametrize("spare", [60, 300])
def test_nan_scores_select_exactly_topk(form, where, spare):
    """NaN scores (an overflowed inner product of a head whose weight is zero) in a list whose topk-th score lies among equal ones at
    the bottom of the range: among so few that an interval of the histogram holds them, or so many that the radix passes decide."""
    dtype, D, n, k = form[:4]
    di = form[4] if len(form) > 4 else 128 if dtype == "bf16" else 64
    rng = np.random.default_rng(n)
    a = rng.integers(1, 200, n).astype(np.float32)
    zero = rng.permutation(n)[: n - k + spare]                  # relu leaves nothing of them: the topk-th score is theirs
    a[zero] = -1
    ik, tree_ik = np.zeros((n, di), np.float32), np.zeros(di, np.float32)
    ik[:, 0] = a
    scores, tree_score = np.maximum(a, 0).astype(np.float64), 0.0
    if where == "committed":
        ik[zero[:3], 1] = 1e38
        scores[zero[:3]] = np.nan
    else:
        tree_ik[1] = 1e38
        tree_score = np.nan
    HI = 2
    iq = np.zeros((D, HI, di), np.float32)
    iq[:, 0, 0], iq[:, 1, 1] = 1, 3e38
    iw = np.zeros((D, HI), np.float32)
    iw[:, 0] = 2.0 ** np.arange(D)
    _check(_select(form, HI, ik, tree_ik, iq, iw), form, scores, tree_score)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("sign", [1, -1])
def test_closed_entries_beyond_the_range_of_the_committed(form, sign):
    """Entries closed inside the tree score far above or far below every committed entry, whose range the histogram may be laid over; at
    the threshold committed entries tie."""
    dtype, D, n, k = form[:4]
    di = form[4] if len(form) > 4 else 128 if dtype == "bf16" else 64
    rng = np.random.default_rng(n + 2)
    ik, tree_ik = np.zeros((n, di), np.float32), np.zeros(di, np.float32)
    ik[:, 0], tree_ik[1] = rng.integers(1, 200, n), 4096
    iq = np.zeros((D, 2, di), np.float32)
    iq[:, 0, 0], iq[:, 1, 1] = 1, 1
    iw = np.zeros((D, 2), np.float32)
    iw[:, 0], iw[:, 1] = 1, sign
    _check(_select(form, 2, ik, tree_ik, iq, iw), form, ik[:, 0].astype(np.float64), 4096.0 * sign)


@pytest.mark.parametrize("form", FORMS)
def test_zeros_of_either_sign_tie(form):
    """All heads of negative weight: the best score is a zero, negative where a product of the two leaves it, positive for an entry
    closed inside the tree.  They tie, and the lower indices win: the committed ones."""
    dtype, D, n, k = form[:4]
    di = form[4] if len(form) > 4 else 128 if dtype == "bf16" else 64
    rng = np.random.default_rng(n + 1)
    HI = 4
    ik = np.zeros((n, di), np.float32)
    ik[:, :HI] = -rng.integers(1, 100, (n, HI))
    worse = rng.permutation(n)[: (n - k) // 2]               # the others, more than topk, all score zero
    ik[worse, 2] = rng.integers(1, 100, len(worse))
    iq = np.zeros((D, HI, di), np.float32)
    iq[:, range(HI), range(HI)] = 1
    iw = np.full((D, HI), -1, np.float32)
    _check(_select(form, HI, ik, np.zeros(di, np.float32), iq, iw), form, -np.maximum(ik, 0).max(1).astype(np.float64), 0.0)


@pytest.mark.parametrize("form", FORMS + [("bf16", 4, 2500, 2400)])
def test_no_room_for_closed_entries_selects_nothing(form):
    """A sequence whose slab cannot hold what its tree may close is flagged by every form, the scoring kernels among them: none of its
    rows are read beyond what it says it has, and its lists are empty."""
    from paper_2609_24698_b200 import binding as tsv
    dtype, D, n, k = form[:4]
    di = form[4] if len(form) > 4 else 128 if dtype == "bf16" else 64
    HI = 8 if D == 4 else 2
    ones = np.ones((D, HI, di), np.float32)
    got = _select(form, HI, np.ones((n, di), np.float32), np.zeros(di, np.float32), ones, ones[:, :, 0], cap=n, status=tsv.ST_CSA_CAP)
    assert (got == -1).all()


# The tcgen05 scoring kernel takes the lists that are left to it: eight heads with up to four nodes, and, of fewer heads, capacities
# beyond the clusters' (room: a list that is short in a cache sized for 450 k entries).  Lists at the edges of its tiles of 128 entries
# and CTAs of four of them; selected by a cluster of CTAs per node, or by one that reads the scores again in every pass.
@pytest.mark.parametrize("D,HI,room", [(4, 8, None), (1, 8, None), (8, 1, 900_000), (8, 4, 900_000), (7, 2, 900_000), (3, 8, 900_000)])
@pytest.mark.parametrize("n", [129, 511, 513, 2688])
def test_tensor_core_scores(D, HI, room, n):
    rng = np.random.default_rng(n + D)
    ik = rng.integers(-3, 4, (n, 128)).astype(np.float32)    # (small integers: exact in bf16, their sums exact in fp32)
    iq = rng.integers(-2, 3, (D, HI, 128)).astype(np.float32)
    iw = rng.integers(1, 4, (D, HI)).astype(np.float32)
    form = ("bf16", D, n, n // 3)
    got = _select(form, HI, ik, np.zeros(128, np.float32), iq, iw, room=room or 5000 + 2 * n)
    scores = np.einsum("dhe,dh->de", np.maximum(np.einsum("ed,nhd->nhe", ik, iq), 0), iw)
    for node in range(D):
        _check(got[node:node + 1], form, scores[node], np.full(node // 2, 0.0))
