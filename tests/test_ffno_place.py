"""Which buffers the factorised surrogate's kernels touch where they are: only
memory of their own device and managed memory.  Another device's pages need not
be mapped, so its memory is copied (host code, compiled here without a GPU)."""
import os
import shutil
import subprocess

import pytest

from paper_2606_16765_gb300 import _build

SRC = r"""
#include <cstdio>
#include "ffno_place.h"
int main()
{
    const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged};
    for (int owner = 0; owner < 3; ++owner)
        for (cudaMemoryType t : types) {
            cudaPointerAttributes at{};
            at.type = t;
            at.device = owner;
            std::printf("%d %d %d\n", owner, (int)t, (int)ffno::place_of(at, 1));
        }
}
"""


def test_only_own_memory_is_used_in_place(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    (tmp_path / "t.cc").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run([gxx, "-std=c++17", "-I", _build.CSRC, "-I", cuda, str(tmp_path / "t.cc"), "-o", exe], check=True)
    rows = [tuple(map(int, l.split())) for l in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines()]
    host, elsewhere, here = 0, 1, 2
    want = {0: host, 1: host, 3: here}                    # unregistered, pinned, managed
    assert len(rows) == 12
    for owner, kind, place in rows:
        assert place == (want[kind] if kind != 2 else here if owner == 1 else elsewhere), (owner, kind, place)
