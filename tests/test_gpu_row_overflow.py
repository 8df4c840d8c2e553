"""One row's scores overflow (finite query, finite keys, products of -inf or +inf): no other row of its warp changes, and where scores are
left, the row is the softmax over them.  On the tensor-core path, whose warps hold 32 rows and read tensor memory together."""
import pytest
import torch

from paper_2609_24698_b200 import synth

pytestmark = pytest.mark.gpu
D, H, TOPK, WINDOW, NODE, HEAD = 5, 64, 700, 128, 2, 5


# room: tokens the capacities are for; the larger ones take the instantiation for long lists.  keys: the window rows whose product with
# the row's query overflows: the first 32 rows each of the two warps sees, or all of them (then every score of the row that is not of
# the tree or an entry)
@pytest.mark.parametrize("L,room", [(128, 140), (128, 6000), (2432, 2450), (2432, 6000)])
@pytest.mark.parametrize("sign,keys", [(-1, "first"), (-1, "window"), (-1, "all"), (1, "first")])
def test_other_rows_are_untouched(L, room, sign, keys):
    from paper_2609_24698_b200 import harness as hz
    sh = synth.Shape("bf16", 1, D, H, 512, 4, TOPK, 2, 128, 128, WINDOW)
    ccap, hcap = hz.capacities(sh, [L], 2 * D)
    eng = hz.VerifyEngine(sh, 1, ccap, hcap, room)
    gen = torch.Generator(device="cuda").manual_seed(L)
    c, inp = eng.caches[0], hz.InputSet.empty(sh, 1)
    nd = inp.layers[0]
    for t in (c.csa_kv, c.csa_ik, c.hca_kv, c.win_kv, nd.q, nd.kv, nd.c_csa, nd.c_hca, nd.ikc, nd.iq, nd.iw, nd.g_csa, nd.g_hca):
        t.normal_(0.0, 0.3, generator=gen)
    c.L.fill_(L)
    nd.parent.copy_(torch.arange(-1, D - 1).view(1, D)); nd.n_nodes.fill_(D)
    # column 0 belongs to the row under test: zero in all other queries, and in all keys but those that overflow
    rows = {"first": list(range(32)) + list(range(64, 96)), "window": list(range(WINDOW)), "all": list(range(WINDOW))}[keys]
    nd.q[..., 0] = 0
    for t in (c.csa_kv, c.hca_kv, c.win_kv, nd.kv):
        t[..., 0] = 1e3 if keys == "all" else 0
    win = c.win_kv.view(WINDOW, 512)
    win[rows, 0] = 1e3
    nd.q[0, NODE, HEAD] = 0
    eng.launch_cycle(inp, refresh=False)
    want = eng.out[0].clone()
    nd.q[0, NODE, HEAD, 0] = sign * 3e38
    eng.launch_cycle(inp, refresh=False)
    torch.cuda.synchronize()
    assert int(eng.status.sum()) == 0
    got = eng.out[0].clone()
    row = got[0, NODE, HEAD].double().clone()
    got[0, NODE, HEAD] = want[0, NODE, HEAD]
    assert torch.equal(got, want) and float(want.abs().max()) > 0
    if sign < 0:
        # visible: the window but its NODE + 1 oldest positions (L is a multiple of the window: slot order), all entries (no block
        # closes at a strict ancestor of the node: positions L and L + 1), the node and its ancestors; all scores left are zero
        k = torch.cat([win[NODE + 1:], c.csa_kv.view(-1, 512)[:L // 4], c.hca_kv.view(-1, 512)[:L // 128], nd.kv[0, :NODE + 1]]).double()
        k = k[k[:, 0] == 0]
        ref = k.mean(0) if len(k) else torch.zeros(512, dtype=torch.float64, device="cuda")
        # (half a unit of bf16 for the result; the weights are equal and exact)
        assert float((row - ref).abs().max()) <= 2.0 ** -8 * float(ref.abs().max()) + 1e-6
