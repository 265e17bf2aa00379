"""Registers of level updates as the compiler reports them: these instances hold
their populations in registers; at a tighter launch bound, or with the code of
rarer nodes compiled in, they spilled and lost 2 to 5 % of a step."""
import re
import subprocess

import pytest

from paper_2004_11863_gb300 import build

UPDATES = [
    "k_stream_collide_x2<D3Q19, float, 0, 0, false, false, NoEdge<D3Q19>>",
    "k_stream_collide_x2<D3Q19, float, 0, 0, true, false, NoEdge<D3Q19>>",
    "k_stream_collide_x2<D3Q19, float, 0, 0, true, true, NoEdge<D3Q19>>",
    "k_stream_collide<D2Q9, 2, float, 0, false, NoEdge<D2Q9>>",
    "k_stream_collide<D2Q9, 2, float, 0, false, EdgeCount>",
    "k_stream_collide<D2Q9, 2, float, 1, true, EdgeCount>",
    "k_stream_collide_pair<D2Q9, 2, 0, true, EdgeCount>",
]


def test_updates_do_not_spill(tmp_path):
    try:
        nvcc = build._nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    src = tmp_path / "updates.cu"
    src.write_text('#include "kernels.cuh"\nusing namespace mlbm;\nvoid* updates[] = {\n'
                   + "".join(f"  (void*){u},\n" for u in UPDATES) + "};\n")
    r = subprocess.run([nvcc, *build.ARCH, *build.FLAGS, f"-I{build.CSRC}", "-Xptxas", "-v",
                        "-c", str(src), "-o", str(tmp_path / "updates.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    # (one more entry per kernel of the header that is no template)
    spills = re.findall(r"Compiling entry function '(\S*stream_collide\S*)'.*?"
                        r"(\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr, re.S)
    assert len(spills) == len(UPDATES)
    assert [s for s in spills if s[1:] != ("0", "0")] == []
