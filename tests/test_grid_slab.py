"""Room for the accepted draws of a warp of the grid form.  A warp keeps them in
a slab until the end of its chunk.  The chunk's indices are taken in tiles of
128, 32 rows to a warp, and a chunk that crosses a multiple of 2^32 in two parts
that each begin with a tile of their own.  Every split of a full chunk has to
fit the slab when every proposal is accepted."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2411_16952_gb300", "csrc")


def _constants(tmp_path):
    cuda = "/usr/local/cuda/include"
    if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")) or shutil.which("g++") is None:
        pytest.skip("no CUDA headers or no host compiler")
    src = tmp_path / "slab.cpp"
    src.write_text('#include <cstdio>\n#include "tkdv_internal.h"\n'
                   'int main() { std::printf("%u %u\\n", tkdv::kAcceptSlab, tkdv::kChunkPerThread); }\n')
    exe = tmp_path / "slab"
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I", cuda, str(src), "-o",
                    str(exe)], check=True)
    return map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())


def _rows(part, warp):
    """Rows of one warp in a part of `part` proposals."""
    tiles = np.arange((part + 127) // 128)
    return int(np.clip(part - 128 * tiles - 32 * warp, 0, 32).sum())


def test_slab_holds_every_split_of_a_full_chunk(tmp_path):
    slab, per_thread = _constants(tmp_path)
    chunk = 128 * per_thread
    worst = max(_rows(a, w) + _rows(chunk - a, w) for a in range(chunk + 1) for w in range(4))
    assert worst <= slab, (worst, slab)
