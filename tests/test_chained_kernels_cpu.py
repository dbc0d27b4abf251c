"""Kernels launched with launch_chained exist before the kernel in front of them has
ended.  Read from the sources: each one waits (chain_begin) before it touches memory,
and neither it nor the helpers it shares read through the read-only path (__ldg, or a
__restrict__ parameter), which is for data that nobody writes while the kernel exists."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1608_01362_gb300", "csrc")
HELPERS = ("carry_runs.cuh", "gather.cuh", "ranges.cuh", "rowwalk.cuh", "seg_gather.cuh",
           "staged_stream.cuh", "update.cuh")


def _sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
        out[os.path.basename(path)] = re.sub(r"//[^\n]*", "", text)
    return out


def _close(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def _kernels(sources):
    """name -> (parameters, body) of every __global__ function"""
    out = {}
    for text in sources.values():
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*(\())?", text):
            at = _close(text, m.start(1), "()") + 1 if m.group(1) else m.end()
            name = re.compile(r"\s*(\w+)\s*\(").match(text, at)
            end = _close(text, name.end() - 1, "()")
            body = text.index("{", end)
            out[name.group(1)] = (text[name.end():end], text[body + 1:_close(text, body, "{}")])
    return out


def _chained(sources):
    names = set()
    for text in sources.values():
        for m in re.finditer(r"\blaunch_chained\(", text):
            call = text[m.end():_close(text, m.end() - 1, "()")]
            if call.startswith("void (*kernel)"):
                continue  # its definition
            first = re.split(r",(?![^<]*>)", call.replace("->", "."))[0]
            found = re.findall(r"\w+_kernel\b", first)
            if not found:  # a variable: what was assigned to it last
                var = first.strip()
                found = re.findall(r"\w+_kernel\b", re.findall(
                    r"auto %s =([^;]*);" % re.escape(var), text[:m.start()])[-1])
            assert found, call
            names.update(found)
    return names


def test_chained_kernels_wait_first():
    sources = _sources()
    kernels, chained = _kernels(sources), _chained(sources)
    assert len(chained) >= 25
    waiting = {n for n, (_, body) in kernels.items() if "chain_begin()" in body}
    assert chained <= waiting, chained - waiting
    for name in sorted(waiting):
        before = kernels[name][1].split("if (!chain_begin()) return;")
        assert len(before) == 2, name
        rest = re.sub(r"(extern )?__shared__[^;]*;", "", before[0])  # declarations are no access
        assert not re.search(r"\[|->|__ld|atomic|= \*", rest), (name, rest)


def test_chained_kernels_read_plainly():
    sources = _sources()
    for name, (params, body) in sorted(_kernels(sources).items()):
        if "chain_begin()" in body:
            assert "__restrict__" not in params, name
            assert "__ldg" not in body, name
    for name, text in sources.items():
        if name in HELPERS or "launch_chained(" in text and name != "common.cuh":
            text = text.replace("CHAINED ? __ldca(p) : __ldg(p)", "")
            assert "DenseWalk" not in text or name == "bc.cu" or "int32_t, true> w;" in text
            for m in re.finditer(r"__ldg|ld\.global\.nc", text):
                # only in kernels that are launched one after the other
                start = text.rfind("__global__", 0, m.start())
                assert start >= 0 and "chain_begin()" not in text[start:m.start()] and \
                    m.start() < _close(text, text.index("{", start), "{}"), (name, m.group())
