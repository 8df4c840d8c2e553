"""What the library keeps between calls on the host."""
import os
import struct


def _tls_bytes(path):
    """Size of the thread-local storage an ELF64 file asks for (program header PT_TLS)."""
    data = open(path, "rb").read()
    phoff, = struct.unpack_from("<Q", data, 32)
    phentsize, phnum = struct.unpack_from("<HH", data, 54)
    for i in range(phnum):
        kind, = struct.unpack_from("<I", data, phoff + i * phentsize)
        if kind == 7:
            return struct.unpack_from("<Q", data, phoff + i * phentsize + 40)[0]
    return 0


def test_library_keeps_no_tables_per_thread():
    """Thread-local storage of a library loaded at run time is allocated on a thread's first use of it: the library, which allocates
    nothing, has next to none (tensor maps were kept there once, 90 KB, found again by the addresses of a call's inputs)."""
    from paper_2609_24698_b200.build import build_library
    assert _tls_bytes(build_library()) <= 4096


def test_every_exported_call_is_declared():
    """What a caller can reach stands in tsv.h, but for the benchmark's stage timer."""
    import subprocess
    from paper_2609_24698_b200.build import build_library
    from tests.test_abi import declared_functions
    out = subprocess.run(["nm", "-D", "--defined-only", build_library()], capture_output=True, text=True, check=True).stdout
    exported = {line.split()[-1] for line in out.splitlines() if " T " in line}
    c_names = {n for n in exported if not n.startswith("_")}
    assert c_names - set(declared_functions()) == {"tsv_bench_tree_verify_attn_stages"}


def test_cycle_driver_passes_the_tensors_of_the_moment(monkeypatch):
    """The structs launch_cycle keeps follow the engine's caches and scratch pads; those of the inputs are the given set's."""
    import ctypes as C
    import torch
    from paper_2609_24698_b200 import binding as tsv, harness as hz, synth
    sh = synth.Shape("fp32", 2, 5, 4, 16, 2, 4, 1, 8, 4, 8)
    eng = hz.VerifyEngine(sh, 2, [8, 8], [4, 4], 32, device="cpu")
    seen = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: None)
    monkeypatch.setattr(tsv, "tree_verify_layer", lambda shape, cache, nodes, scratch, *a: seen.append((cache.csa_kv, nodes.q, scratch.hca_s)))

    def refresh(shape, pack, *a):
        for l in range(pack.n):
            c, n, s = [C.cast(x[l], C.POINTER(t)).contents for x, t in ((pack.caches, tsv.CCache), (pack.nodes, tsv.CNodes), (pack.scratch, tsv.CScratch))]
            assert seen[l] == (c.csa_kv, n.q, s.hca_s)
    monkeypatch.setattr(tsv, "accept_and_refresh", refresh)
    sets = [hz.InputSet.empty(sh, 2, "cpu") for _ in range(2)]
    for step in range(5):
        if step == 2:
            eng.caches[1].csa_kv = eng.caches[1].csa_kv.clone()
        if step == 3:
            eng.scratch[0].hca_s.data = eng.scratch[0].hca_s.clone()
        if step == 4:
            eng.caches[0] = eng.caches[0].clone()
        inp = sets[step % 2]
        seen.clear()
        eng.launch_cycle(inp)
        assert seen == [(eng.caches[l].csa_kv.data_ptr(), inp.layers[l].q.data_ptr(), eng.scratch[l].hca_s.data_ptr()) for l in range(2)]
