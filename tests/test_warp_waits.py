"""In the tensor-core kernels, a role that a whole warp runs must not let a single lane
leave a wait while the others go on to instructions that the warp executes together.
Read from the sources (a wait that runs out is not provoked on a GPU): in a role with
such instructions between its waits, every condition on a barrier or on the abort flag
is the warp's vote."""
from __future__ import annotations

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_06452_gb300", "csrc")
ROLE = re.compile(r"^    (?:\} else )?if \((warp\b[^{]*)\) \{ // ----.*$", re.M)


def _whole_warp_roles(src):
    """The bodies of the roles whose condition leaves all 32 lanes in."""
    heads = list(ROLE.finditer(src))
    for h in heads:
        if "lane == 0" in h.group(1):
            continue
        yield h.group(0).strip(), src[h.end():src.index("\n    }", h.end())]


def _arguments(body, name):
    """The text inside each call of `name`."""
    for m in re.finditer(re.escape(name) + r"\(", body):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(body[i], 0)
            i += 1
        yield m.start(), i


@pytest.mark.parametrize("file,roles", [("mlp_gemm.cu", 2), ("mlp_infer.cu", 3), ("mlp_train.cu", 2)])
def test_waits_of_whole_warps_are_voted_on(file, roles):
    with open(os.path.join(CSRC, file)) as f:
        src = f.read()
    found = list(_whole_warp_roles(src))
    assert len(found) == roles, [h for h, _ in found]
    for head, body in found:
        first = re.search(r"mbar_wait", body).start()
        together = re.findall(r"tmem_ld\w*\(|__\w+_sync\(|__syncwarp\(|elect_one\(|warp_ok\(", body[first:])
        if together == ["__syncwarp("] and body.rstrip().endswith("__syncwarp();"):
            continue  # the lanes meet again only at the end
        voted = list(_arguments(body, "warp_ok"))
        assert voted, head
        for m in re.finditer(r"(?:tc::mbar_wait(?:_cluster)?\(|\*abort_flag(?!\s*=[^=]))", body):
            if any(a < m.start() < b for a, b in voted):
                continue
            statement = re.sub(r"//[^\n]*", "", body[:m.start()])
            statement = statement[max(statement.rfind(c) for c in ";{}") + 1:].strip()
            # kept for a vote further on, or one lane's wait on work it has issued, whose outcome is not used
            later = re.fullmatch(r"(?:bool )?ok =.*", statement, re.S) and "warp_ok(ok)" in body[m.end():]
            assert later or statement in ("", "if (zload)"), (head, statement, body[m.start():m.end() + 60])
        # nothing leaves a step on one lane's outcome but by way of the vote
        for m in re.finditer(r"if \(!ok\) (?:break|return)", body):
            assert "warp_ok(ok)" in body[m.end():] or "ok = tc::warp_ok(ok);" in body[m.start() - 60:m.start()], head
