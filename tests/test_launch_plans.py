"""The engine's launch plans and workspace sizes for a configuration, computed without a GPU by a
small program around the engine's own source (plan_probe.cu)."""
import json
import os
import subprocess

import pytest

from paper_2607_12287_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))
SEL_THRESHOLD, SEL_TOPK = 0, 1


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    lib = b.build()
    exe = str(tmp_path_factory.mktemp("probe") / "plan_probe")
    subprocess.run([b.NVCC, *b.ARCH, "-O1", "-std=c++17", "-I", os.path.join(b.ROOT, "include"),
                    os.path.join(HERE, "plan_probe.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", exe],
                   check=True, capture_output=True)

    def run(tokens, dim, heads, mlp, views=1, select=SEL_THRESHOLD, topk=0, mlp_tokens=0):
        args = map(str, (tokens, dim, heads, mlp, views, select, topk, mlp_tokens))
        return json.loads(subprocess.run([exe, *args], check=True, capture_output=True, text=True).stdout)

    return run


def scratch_of(plan, dim, rows):
    """fp32 values of the partial tiles that one launch writes: [tile][split][rows of a tile][128]."""
    return -(-dim // 128) * -(-rows // plan["bn"]) * plan["splits"] * plan["bn"] * 128 if plan["defer"] else 0


@pytest.mark.parametrize("tokens,dim,heads,mlp,views", [(256, 1152, 16, 4304, 1), (256, 1152, 16, 4304, 3), (196, 192, 3, 768, 6),
                                                       (1024, 1152, 16, 4304, 32), (256, 2048, 16, 8192, 1),
                                                       (324, 768, 12, 3072, 4), (64, 512, 8, 2048, 2)])
@pytest.mark.parametrize("select,topk", [(SEL_THRESHOLD, 0), (SEL_TOPK, 10), (SEL_TOPK, 100)], ids=["threshold", "top10", "top100"])
def test_split_scratch_holds_every_row(probe, tokens, dim, heads, mlp, views, select, topk):
    # (top-k selects NaN scores beside its k lowest: any plan may meet any number of rows)
    p = probe(tokens, dim, heads, mlp, views, select, topk)
    rows = tokens * views
    plans = [pl for name, group in p.items() if name.startswith(("full", "inc", "band")) and name != "bands" for pl in group]
    need = max(scratch_of(pl, dim, rows) for pl in plans)
    assert need <= p["scratch"]
    assert p["bands"][-1] == rows or len(p["bands"]) == 1
