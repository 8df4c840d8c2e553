"""The refresh for every layer count at which its form changes (one cluster kernel, two kernels, several launches), and the host arrays
of a cycle following the objects they were built from."""
import pytest
import torch

from paper_2609_24698_b200 import synth


@pytest.mark.gpu
@pytest.mark.parametrize("layers", [1, 8, 9, 13])
def test_refresh_layer_counts(layers):
    from tests.test_gpu_parity import lockstep
    cfg = synth.small_config(name=f"layers{layers}", dtype="bf16", B=3, D=5, H=4, d=16, m_csa=2, topk=6, HI=1, di=8, m_hca=4, window=8,
                             L_min=3, L_max=30, layers=layers, seed=60 + layers, cfg_id=212, p=0.9)
    lockstep(cfg, cycles=3, check_recompress="final")


def test_layer_pack_follows_its_objects():
    from paper_2609_24698_b200 import binding as tsv, harness as hz
    sh = synth.Shape("fp32", 2, 5, 4, 16, 2, 4, 1, 8, 4, 8)
    caches = [tsv.alloc_cache(sh, [8, 8], [4, 4], "cpu")]
    scratch, inp = [tsv.alloc_scratch(sh, "cpu")], hz.InputSet.empty(sh, 1, "cpu")
    pack = tsv.LayerPack(caches, inp.layers, scratch)
    assert pack.current(caches, inp.layers, scratch)
    caches[0].csa_kv = caches[0].csa_kv.clone()                     # a field assigned
    assert not pack.current(caches, inp.layers, scratch)
    pack = tsv.LayerPack(caches, inp.layers, scratch)
    inp.layers[0].q.data = inp.layers[0].q.clone()                  # a storage exchanged in place
    assert not pack.current(caches, inp.layers, scratch)
    pack = tsv.LayerPack(caches, inp.layers, scratch)
    assert not pack.current(caches, inp.layers, [tsv.alloc_scratch(sh, "cpu")])      # another object


def test_layer_pack_notices_an_object_at_the_address_of_another():
    from paper_2609_24698_b200 import binding as tsv, harness as hz
    sh = synth.Shape("fp32", 2, 5, 4, 16, 2, 4, 1, 8, 4, 8)
    scratch, inp = [tsv.alloc_scratch(sh, "cpu")], hz.InputSet.empty(sh, 1, "cpu")
    caches = [tsv.alloc_cache(sh, [8, 8], [4, 4], "cpu")]
    for _ in range(20):
        pack = tsv.LayerPack(caches, inp.layers, scratch)
        tensors = {n: getattr(caches[0], n).clone() for n in tsv.CACHE_TENSORS}
        caches.clear()
        caches.append(tsv.LayerCache(**tensors))             # (takes the place the allocator has just got back)
        assert not pack.current(caches, inp.layers, scratch)
