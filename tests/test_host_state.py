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
