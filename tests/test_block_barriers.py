"""Barriers between warp 0's stores of a pending self-served request and the block's reads
of it (no GPU: the order of accesses in the source of gread_impl).

Warp 0 stores the request while it acquires a page and while it checks the page's readahead
mark; every thread of the block reads whether one is pending.  A store and a read with no
barrier of the whole block between them race: warps would disagree on whether the block
copies a request, and meet different barriers."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_05366_gb300", "csrc",
                   "gfs_device.cuh")


def _body(src, name):
    """The braces' content of the definition of function `name` (the last one in the file)."""
    at = [m.start() for m in re.finditer(r"\b%s\(" % name, src)]
    for a in reversed(at):
        brace, semi = src.find("{", a), src.find(";", a)
        if 0 <= brace < semi:
            depth, i = 0, brace
            while True:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
                if depth == 0:
                    return src[brace + 1:i - 1]
    raise AssertionError("no definition of " + name)


def _accesses(src):
    """'W' (store by warp 0), 'R' (read by every thread), 'B' (barrier on every path) in program order."""
    loop = _body(src, "gread_impl")
    loop = loop[loop.index("for (unsigned long long p = p0"):]
    loop = loop[loop.index("{") + 1:loop.rindex("++p;")]
    serves = {f: "self_job()" in _body(src, f).split("return", 1)[0] for f in ("block_self_serve", "block_serve_arriving")}
    out, depth = [], 0
    token = re.compile(r"[{}]|__syncthreads\(\)|self_job\(\)\.n = |self_job\(\)|acquire_begin\(|check_mark\(|"
                       r"block_self_serve\(|block_serve_arriving\(")
    for m in token.finditer(loop):
        t = m.group().rstrip("(")
        if t in "{}":
            depth += 1 if t == "{" else -1
        elif t == "__syncthreads()":
            if depth == 0:  # a barrier under a condition does not count
                out.append("B")
        elif t in ("acquire_begin", "check_mark", "self_job().n = "):
            out.append("W")
        elif t == "self_job()" or serves[t]:
            out.append("R")
    return out


def test_pending_request_is_read_between_barriers():
    with open(SRC) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    acc = _accesses(src)
    assert acc.count("W") >= 3 and acc.count("R") >= 2
    last = None
    for a in acc + acc:  # two turns of the loop
        if a == "B":
            last = None
            continue
        assert last in (None, a), "".join(acc)
        last = a
