"""A kernel that starts before its predecessor in the stream has ended is
resident while that predecessor writes the populations, moments and multipliers
it will read.  CUDA's non-coherent load (__ldg, or what the compiler makes of a
const __restrict__ parameter) is only for data that is read-only for a kernel's
whole lifetime, and a __restrict__ load may move above the wait.  No run shows
such a fault reliably, so the sources are read: every kernel that starts early,
and every device function it reaches."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_1903_01111_gb300" / "csrc"

# written by the host alone, before any launch
TABLES = {"recs", "qv", "uwv", "wqv", "wq", "wbody", "runs", "dp", "next"}
# written by the kernel; read back, if at all, by the thread that wrote
OUTPUTS = {"fout", "ok", "mom", "mom_out", "lam_out", "o"}


def _functions(text):
    """name -> (is a kernel, source from its qualifier to its closing brace)."""
    text = re.sub(r"//[^\n]*", "", text)
    out = {}
    for m in re.finditer(r"__(global|device)__[^;{}]*?\b(\w+)\((?=[^;{}]*\)\s*\{)", text):
        sig = text[m.start():text.index("{", m.end())]
        name = re.sub(r"__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", sig)
        name = re.search(r"(\w+)\s*\(", name.replace("__forceinline__", "").split("void", 1)[-1]) or m
        end, depth = text.index("{", m.end()), 0
        for i in range(end, len(text)):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            if depth == 0:
                break
        key = name.group(1) if name is not m else m.group(2)
        out[key] = (m.group(1) == "global", out.get(key, (0, ""))[1] + text[m.start():i + 1])
    return out


def _early():
    fns = {}
    for f in ("kernels.cuh", "adjoint.cuh"):
        fns.update(_functions((CSRC / f).read_text()))
    kernels = set()
    for f in ("kernels.cuh", "adjoint.cuh"):
        kernels |= set(re.findall(r"launch_early\((k_\w+)", (CSRC / f).read_text()))
    reached, todo = set(), list(kernels)
    while todo:
        n = todo.pop()
        if n in reached:
            continue
        reached.add(n)
        todo += [c for c in fns if c not in reached and re.search(rf"\b{c}\s*(<[^;(){{}}]*>)?\(", fns[n][1])]
    return fns, kernels, reached


def test_every_early_kernel_is_found_and_waits():
    fns, kernels, reached = _early()
    assert {"k_bulk", "k_bulk_list", "k_bulk_seq", "k_links", "k_fused", "k_inline", "k_adj_bulk", "k_adj_pair",
            "k_adj_links", "k_adj_links_open"} == kernels
    assert {"pull_node", "pair_pull", "eval_link", "adj_link", "adj_open_row", "open_ends", "fill_inlet"} <= reached
    for k in kernels:
        calls = {c for c in reached if re.search(rf"\b{c}\s*(<[^;(){{}}]*>)?\(", fns[k][1])}
        text = fns[k][1] + "".join(fns[c][1] for c in calls)
        assert "wait_for_previous()" in text and "let_next_start()" in text, k


@pytest.mark.parametrize("what", ["__ldg", "__restrict__"])
def test_early_kernels_load_what_others_write_coherently(what):
    fns, _, reached = _early()
    wrong = []
    for n in sorted(reached):
        body = fns[n][1]
        if what == "__ldg":
            for a in re.findall(r"__ldg\(([^;]*)", body):
                if not re.match(r"(&?(lay|fl)\.|&recs\[|\(const uint2\*\)\(lay\.word)", a):
                    wrong.append((n, a[:40]))
        else:
            for decl in re.findall(r"([\w:<> ]+)\*\s*__restrict__\s+(\w+)", body):
                if decl[1] not in (TABLES if decl[0].strip().startswith("const") else OUTPUTS):
                    wrong.append((n, decl[1]))
    assert not wrong, wrong


def test_no_population_is_accessed_through_another_type():
    """A pair of floats stored as one 64-bit integer and read back as a float by
    the same thread (the open node beside it) is undefined: the compiler may take
    the two for different objects and move the load above the store."""
    for f in ("kernels.cuh", "adjoint.cuh", "pair32.cuh"):
        text = re.sub(r"//[^\n]*", "", (CSRC / f).read_text())
        assert not re.search(r"\*\s*\(\s*(const )?(unsigned long long|uint64_t|double|int64_t)\s*\*\s*\)", text), f
