"""The record of a tile (what the tile plan leaves for the attention and merge kernels), packed and unpacked by the functions the kernels
use, compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <stdio.h>
#include "tc_common.cuh"
using namespace tsv; using namespace tsv::tc;
int main() {
  long long b, tile, mode, nk, general, split, chmax, f32;
  while (scanf("%lld %lld %lld %lld %lld %lld %lld %lld", &b, &tile, &mode, &nk, &general, &split, &chmax, &f32) == 8) {
    TvaPlan p = {};
    p.tc_general = (int)general; p.tc_split = (int)split; p.tc_chmax = (int)chmax; p.tc_f32 = (int)f32;
    const int4 r = tile_record(p, (int)b, (int)tile, (int)mode, (int)nk);
    printf("%d %d %d %d %d %d %d %d %d %d\n", r.x, rec_tile(r), r.z, (int)rec_gather(r), (int)rec_f32(r), rec_chunks(r), rec_chunks_or_many(r), rec_chunk_keys(r), rec_lds(r), rec_items(r));
  }
}
"""


@pytest.fixture(scope="module")
def records(tmp_path_factory):
    d = tmp_path_factory.mktemp("record")
    src, exe = d / "record.cu", d / "record"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2609_24698_b200", "csrc"), "-o", str(exe), str(src)], check=True, capture_output=True)

    def run(rows):
        out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, r)) for r in rows), text=True, capture_output=True, check=True).stdout
        return [list(map(int, line.split())) for line in out.splitlines()]
    return run


def test_every_field_comes_back(records):
    """Chunks up to the longest lists a shape may ask for (2^30 tokens, an entry each), sequences up to a grid's, tiles up to the
    largest tree's; the chunks of a tile cover its keys."""
    chunk = 512
    keys = [1, 32, 512, 513, 768, 769, 1536, 1537, 4096, 65535 * chunk, 65535 * chunk + 1, 65536 * chunk + 1, 65537 * chunk, 2 ** 30, 2 ** 31 - 1024]
    rows = [(b, tile, mode, nk, general, split, chmax, f32) for b in (0, 65534) for tile in (0, 15, 31) for mode in (1, 2) for nk in keys
            for general, f32 in ((0, 1), (1, 0)) for split, chmax in ((1, 2 ** 22), (37, 37), (74, 74))
            if general or nk <= 1536]
    for (b, tile, mode, nk, general, split, chmax, f32), got in zip(rows, records(rows), strict=True):
        gb, gtile, gnk, gather, gf32, nch, some, stride, lds, items = got
        assert (gb, gtile, gnk, gather) == (b, tile, nk, mode == 2), (nk, got)
        assert 128 <= stride <= 768 and stride % 128 == 0 and (nch - 1) * stride < nk <= nch * stride, (nk, got)
        assert 0 <= lds <= 2 and items == nch << lds <= max(split, nch) and some == min(nch, 65535), (nk, got)
        assert gf32 == (f32 or nk <= 768), (nk, got)
