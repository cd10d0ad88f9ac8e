"""Kernels of a launch chain start while any number of earlier kernels of the stream still run or wait: until chain_wait() they
may use their parameters and shared memory only.  Checked on the sources: a read that comes too early gives wrong results only
when the scheduler happens to make room for it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_11101_b200", "csrc")
# names the kernels give to members of their one parameter structure
ALIASES = {"bv", "pv", "ws", "span", "src", "out_all", "lse"}
# arrays that are part of a parameter structure, not behind a pointer
IN_PARAMETERS = {"inv_freq.turns", "inv_freq.f", "maps.k", "maps.v"}
SCALAR = re.compile(r"^(const\s+)?(unsigned|int|float|double|long long|unsigned long long|size_t|bool)\s+\w+$")


def _closing(text, at):
    """Index behind the bracket that closes the one at `at`."""
    close = {"(": ")", "{": "}"}[text[at]]
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == text[at]) - (text[i] == close)
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced source")


def _kernels():
    """(name, parameters, body) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        for m in re.finditer(r"__global__\s+void\s*", text):
            at = m.end()
            bounds = re.match(r"__launch_bounds__\s*", text[at:])
            if bounds:
                at = _closing(text, at + bounds.end())
            name = re.match(r"\s*(\w+)\s*", text[at:])
            at += name.end()
            end = _closing(text, at)
            params = [re.sub(r"\s+", " ", x).strip() for x in text[at + 1:end - 1].split(",")]
            body_at = text.index("{", end)
            yield name.group(1), params, text[body_at:_closing(text, body_at)]


KERNELS = {name: (params, body) for name, params, body in _kernels()}


def early_reads(params, prologue):
    """What a kernel's text before chain_wait() does that may touch global memory."""
    names = {re.search(r"(\w+)$", x).group(1) for x in params if not SCALAR.match(x)} | ALIASES
    found = re.findall(r"__ldg|ld\.global|ld\.acquire|atomic\w+|cp\.async", prologue)
    prologue = re.sub(r'"[^"]*"', '""', prologue)
    for name in names:
        for m in re.finditer(r"(?<![\w.>])%s((?:\.\w+)*)\s*(->|\[|\(|)" % name, prologue):
            path, after = name + m.group(1), m.group(2)
            if after == "[" and path in IN_PARAMETERS:
                continue
            # indexed, dereferenced, or handed over as a whole (a pointer, or a structure that holds some)
            if after in ("[", "->") or not m.group(1) or re.search(r"(^|[=(,+{;])\s*\*\s*$", prologue[:m.start()]):
                found.append(prologue[m.start():m.end()])
    return found


def test_the_check_sees_early_reads():
    params = ["DecodeArgs a", "const int* __restrict__ rows", "int n"]
    for bad in ("make_line(a, s, n);", "int x = rows[n];", "int x = a.doc_offsets[2];", "int x = *a.status;", "__ldg(p)", "f(rows);"):
        assert early_reads(params, bad), bad
    for good in ("int x = blockIdx.x * n;", "int y = a.n_heads / 2;", "s_sum[threadIdx.x] = n;"):
        assert not early_reads(params, good), good


@pytest.mark.parametrize("name", sorted(n for n, (_, body) in KERNELS.items() if "chain_next()" in body or "chain_wait()" in body))
def test_no_global_memory_before_the_wait(name):
    params, body = KERNELS[name]
    assert body.count("chain_wait()") == 1, "waits once, on every path"
    prologue = body[:body.index("chain_wait()")]
    # CF_PARAMS only names the members of the parameter structure
    assert early_reads(params, prologue.replace("CF_PARAMS;", "")) == []
    assert "return;" not in prologue


def test_every_chained_launch_has_a_waiting_kernel():
    """Whatever goes through launch_chained (or asks for programmatic serialisation itself) waits; the probe does not."""
    waiting = {n for n, (_, body) in KERNELS.items() if "chain_wait()" in body}
    assert waiting | {"wait_probe_kernel"} == set(KERNELS)
