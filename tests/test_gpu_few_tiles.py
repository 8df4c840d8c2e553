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
    (150, 3, 600, [40 + 7 * i for i in range(150)]),          # two or three tiles a pair, all ragged: staged rows under the next item's queries
])
def test_shares_of_columns(B, D, topk, lengths):
    cfg = synth.Config(f"few_{B}_{D}", 217, synth.Shape("bf16", B, D, 64, 512, 2, topk, 2, 128, 16, 128), L_min=1, L_max=max(lengths), layers=1, seed=31 + B)
    lockstep(cfg, cycles=2, lengths=lengths, want_topk=False)


@pytest.mark.parametrize("D,L", [(3, 3000), (5, 400), (8, 1100)])
@pytest.mark.parametrize("room", [600, 6000])
def test_output_aligned_to_sixteen_bytes(D, L, room):
    """An output that starts 16 bytes past a 32-byte boundary gets the same bytes as an aligned one, and nothing around it is written: whole
    tiles and ragged ones, of one chunk and of several, in capacities of either kind."""
    import torch
    from paper_2609_24698_b200 import harness as hz
    sh = synth.Shape("bf16", 1, D, 64, 512, 2, 300, 2, 128, 16, 128)
    ccap, hcap = hz.capacities(sh, [L], 2 * D)
    eng = hz.VerifyEngine(sh, 1, ccap, hcap, max(L + 2 * D, room))
    gen = torch.Generator(device="cuda").manual_seed(D)
    c = eng.caches[0]
    for t in (c.csa_kv, c.csa_ik, c.hca_kv, c.win_kv):
        t.normal_(generator=gen)
    c.L.fill_(L)
    inp = hz.InputSet.empty(sh, 1)
    nd = inp.layers[0]
    for t in (nd.q, nd.kv, nd.c_csa, nd.c_hca, nd.ikc, nd.iq, nd.iw, nd.g_csa, nd.g_hca):
        t.normal_(0.0, 0.05, generator=gen)
    nd.parent.copy_(torch.arange(-1, D - 1).view(1, D)); nd.n_nodes.fill_(D)
    eng.launch_cycle(inp, refresh=False)
    want, n = eng.out[0].clone(), eng.out[0].numel()
    around = torch.full((n + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    assert around.data_ptr() % 32 == 0
    eng.out = [around[24:24 + n].view(want.shape)]
    eng.launch_cycle(inp, refresh=False)
    torch.cuda.synchronize()
    assert int(eng.status.sum()) == 0 and float(want.abs().max()) > 0
    assert torch.equal(eng.out[0], want)
    assert bool((around[:24] == 7).all()) and bool((around[24 + n:] == 7).all())
