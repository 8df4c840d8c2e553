"""branch_state_build followed by tree_verify_attn as two calls, against the oracle: the other tests drive the device through
tree_verify_layer, whose state build also leaves the closed entries where the attention reads them.  Here the tile plan packs them."""
import pytest

from paper_2609_24698_b200 import synth
from tests.test_gpu_parity import lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture
def separate_calls(monkeypatch):
    from paper_2609_24698_b200 import binding as tsv, harness as hz

    def launch_cycle(self, inp, attention=True, refresh=True):
        self.status.zero_()
        for l in range(self.n_layers):
            args = (self.cshape, self.caches[l], inp.layers[l], self.scratch[l])
            tsv.branch_state_build(*args, self.status)
            tsv.tree_verify_attn(*args, self.out[l], self.topk_idx[l], self.workspace, self.status)
        if refresh:
            tsv.accept_and_refresh(self.cshape, self._pack(inp), inp.draft, inp.target, self.accept_len, self.accept_path, self.bonus, self.status)
    monkeypatch.setattr(hz.VerifyEngine, "launch_cycle", launch_cycle)


# D, lengths, topk, layers, page, deferred, lists, graph: short flat stacks; ranked short lists; a sequence cut into chunks; gathered
# tiles; pages; lists over all SMs; trees of more than one CTA pair's nodes
@pytest.mark.parametrize("D,lengths,topk,layers,page,deferred,lists,graph", [
    (8, [0, 3, 255, 700], 512, 3, 0, False, True, False), (6, [2050, 2300, 400], 512, 2, 0, True, False, False), (5, [3900], 512, 2, 0, False, True, True),
    (8, [3000, 4500, 130], 100, 1, 0, False, False, False), (8, [300, 1100, 2500, 3900], 256, 2, 128, False, True, False),
    (7, [34000, 900], 300, 1, 0, False, False, False), (12, [640, 1500], 512, 2, 128, False, False, True)])
def test_tensor_core_shapes(separate_calls, D, lengths, topk, layers, page, deferred, lists, graph):
    from paper_2609_24698_b200 import binding as tsv
    cfg = synth.Config(f"separate_{D}_{topk}", 216, synth.Shape("bf16", len(lengths), D, 64, 512, 4, topk, 4, 128, 128, 128), layers=layers,
                       L_min=0, L_max=max(lengths), seed=D + len(lengths))
    lockstep(cfg, cycles=2, lengths=lengths, page_tokens=page, flags=tsv.FLAG_HCA_DEFERRED if deferred else 0, want_topk=lists, graph=graph)


@pytest.mark.parametrize("dtype,d,di", [("fp32", 128, 64), ("bf16", 64, 32)])
def test_other_shapes(separate_calls, dtype, d, di):
    cfg = synth.Config(f"separate_{dtype}", 217, synth.Shape(dtype, 4, 8, 16, d, 4, 48, 2, di, 32, 40), layers=2, L_min=0, L_max=900, seed=8)
    lockstep(cfg, cycles=2, lengths=[0, 150, 511, 900])


@pytest.mark.parametrize("D,L", [(8, 40000), (12, 3000)])
def test_selections_in_a_row_share_a_workspace(D, L):
    """The selections of two layers without a state build between them, the way the benchmark times that stage: the next one's scores must
    not reach the workspace while the one before still reads its own (scores over all SMs, a cluster per node)."""
    import torch
    from paper_2609_24698_b200 import binding as tsv, harness as hz
    sh = synth.Shape("bf16", 4, D, 64, 512, 4, 512, 4, 128, 128, 128)
    ccap, hcap = hz.capacities(sh, [L] * 4, 2 * D)
    eng = hz.VerifyEngine(sh, 2, ccap, hcap, L + 2 * D, want_topk=True)
    gen = torch.Generator(device="cuda").manual_seed(L)
    inp = hz.InputSet.empty(sh, 2)
    inp.layers[0].parent.copy_(torch.arange(-1, D - 1).expand(4, D)); inp.layers[0].n_nodes.fill_(D)
    for c, nd in zip(eng.caches, inp.layers):
        c.L.fill_(L)
        for t in (c.csa_ik, nd.ikc, nd.iq, nd.iw):
            t.normal_(generator=gen)
    eng.launch_cycle(inp, refresh=False)
    torch.cuda.synchronize()
    want = [t.clone() for t in eng.topk_idx]
    assert int(eng.status.sum()) == 0 and not torch.equal(want[0], want[1])
    for _ in range(20):
        for t in eng.topk_idx:
            t.fill_(-2)
        for l in range(2):
            tsv.bench_tree_verify_attn_stages(eng.cshape, eng.caches[l], inp.layers[l], eng.scratch[l], eng.out[l], eng.topk_idx[l], eng.workspace,
                                              eng.status, tsv.STAGE_SELECT)
        assert all(torch.equal(a, b) for a, b in zip(eng.topk_idx, want))
