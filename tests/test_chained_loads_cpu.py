"""Kernels launched with programmatic serialisation are resident while their
predecessor still writes what they read.  Read-only loads (__ldg, or const pointers
marked __restrict__) are for data that nobody writes while the kernel is resident, and
the compiler may move them, and cache-operator intrinsics, above the wait.  So in the
sources of these kernels only tables fixed long before (twiddles, Green's function)
are read that way, and the wait is each kernel's first statement."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_12629_gb300", "csrc")
TABLES = {"tw", "green"}


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels(text):
    """(name, parameters, body's beginning) of every kernel of a source."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(\w+)\(([^)]*)\)\s*\{", text):
        yield m.group(1), m.group(2), text[m.end():m.end() + 200]


FILES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and "launch_chained(" in _source(f))
CHAINED = [(f, *k) for f in FILES for k in _kernels(_source(f)) if "chain();" in k[2]]


def test_every_chained_launch_waits_first():
    waiting = {c[1] for c in CHAINED}
    launched = set()
    for f in FILES:
        for call in re.findall(r"launch_chained\(ctx->chained,(.*?)ctx->stream", _source(f), flags=re.S):
            launched |= set(re.findall(r"\b(\w+_kernel|fft_\w+)\b", call))
    assert launched and launched <= waiting, launched - waiting
    for f, name, _, body in CHAINED:
        assert body.lstrip().startswith("chain();"), (f, name)


@pytest.mark.parametrize("f,name,params", [c[:3] for c in CHAINED], ids=[c[1] for c in CHAINED])
def test_parameters(f, name, params):
    read_only = {p.split()[-1].lstrip("*") for p in params.split(",") if "const" in p and "__restrict__" in p}
    assert read_only <= TABLES, (f, name, read_only - TABLES)


@pytest.mark.parametrize("f", FILES)
def test_loads(f):
    text = _source(f)
    for arg in re.findall(r"__ldg\(([^;]*)", text):
        assert re.match(r"&(\w+)\[", arg) and re.match(r"&(\w+)\[", arg).group(1) in TABLES, arg[:40]
    assert not re.findall(r"__ld(?:c[agsv]|lu)\(", text)
