"""Source check of the climb's shared copy of the diagonal (no GPU): every lane of
the owner's warp reads q_kk from it, so in one-warp groups, whose reductions hold
no barrier, a sync has to stand between the writes and the first move."""
import pathlib
import re

CORE = (pathlib.Path(__file__).resolve().parents[1] / "paper_1706_00037_gb300" / "csrc" /
        "ascent_core.cuh")


def test_one_warp_groups_sync_after_writing_the_diagonal():
    text = re.sub(r"//[^\n]*", "", CORE.read_text())
    body = text[text.index("ascend_one("):]
    write, moves = body.index("diag[c * T + g] ="), body.index("for (;;)")
    assert write < moves < body.index("reinterpret_cast<const int8_t*>(diag)[k]")
    assert re.search(r"T == 32\)\s*grp\.sync\(\);", body[write:moves])
