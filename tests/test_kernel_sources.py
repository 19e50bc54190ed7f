"""Rules of the CUDA sources that no run can show to be broken without hanging a GPU:
read from the text.  CPU only."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2606_01790_gb300" / "csrc"


def functions(name):
    """{function: body without comments} of the functions of a source file whose
    brace opens on the line of their closing parenthesis."""
    text = re.sub(r"//[^\n]*", "", (CSRC / name).read_text())
    out = {}
    for m in re.finditer(r"^[^\n;{}=]*?\b(\w+)\((?:[^(){};]|\([^()]*\))*\)\s*\{", text, flags=re.M):
        if m.group(1) in ("if", "for", "while", "switch"):
            continue
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out[m.group(1)] = text[m.end():i - 1]
    return out


@pytest.mark.parametrize("helper", ["cluster_sync", "cluster_arrive", "cluster_wait", "named_bar_sync", "tmem_dealloc"])
def test_barriers_that_want_a_converged_warp_converge_it(helper):
    """An aligned barrier has no time limit: reached by a diverged warp it may
    never complete.  Callers have per-lane branches right before these."""
    body = functions("ptx.cuh")[helper]
    assert "__syncwarp();" in body and body.index("__syncwarp();") < body.index("asm")


def test_no_other_source_issues_such_a_barrier_itself():
    for path in sorted(CSRC.glob("*.cu*")):
        if path.name != "ptx.cuh":
            assert not re.search(r'"[^"]*(barrier\.cluster|bar\.sync|tcgen05\.dealloc)', path.read_text()), path.name


@pytest.mark.parametrize("role", ["mma_s_loop", "mma_pv_loop", "softmax_unit", "softmax_loop", "convert_loop"])
def test_warp_wide_attention_roles_leave_together(role):
    """Lanes that read another role's failure flag one by one may disagree, and those
    that stay then wait for the others in the next warp vote for ever.  These
    roles learn of a failure only through warp_wait's vote, at every wait; the
    final wait for their own products is the one that goes on regardless."""
    body = functions("attn.cu")[role]
    assert "abort" not in body
    assert "warp_wait(" in body
    assert re.findall(r"\bmbar_wait\(([^,]*),", body) == (["&ctl->drain"] if role.startswith("mma") else [])


def test_every_attention_wait_sees_another_roles_failure():
    body = functions("attn.cu")["warp_wait"]
    assert body.index("ctl->abort") < body.index("__all_sync(") < body.index("mbar_wait(")


@pytest.mark.parametrize("source,role", [("score.cu", "producer_loop"), ("attn.cu", "k_loader"), ("attn.cu", "v_loader")])
def test_loaders_see_every_copy_land(source, role):
    """A loader that is past its last load when another role gives up still keeps
    the block until its copies are in: they would land in another block's shared
    memory.  The waits for them stand at the function's top level."""
    body = functions(source)[role]
    depth, found = 0, []
    for line in body.split("\n"):
        if "drain_limit(" in line:
            found.append((depth, line))
        depth += line.count("{") - line.count("}")
    assert found and all(d == 0 for d, _ in found)
    assert not re.search(r"if \(ctl->abort\)\s*\{?\s*for", body)
