"""Kernels that may start before their predecessor on the stream has ended (they wait for it by
pdl_wait, or through multi_block) read what that predecessor writes. No pointer among their
parameters may be `const ... __restrict__`, which promises data that nothing writes while the kernel
runs and lets loads take the read-only path; the batch's block tables, written before any launch, may."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2305_18919_gb300", "csrc")
TABLES = {"all", "start"}


def _closing(src, at, pair):
    depth = 0
    for k in range(at, len(src)):
        depth += (src[k] == pair[0]) - (src[k] == pair[1])
        if depth == 0:
            return k
    raise AssertionError("unbalanced source")


def early_kernels():
    """(name, parameters) of every __global__ function that waits for its predecessor."""
    out = []
    for fn in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fn)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__(\())?", src):
            at = m.end() if not m.group(1) else _closing(src, m.start(1), "()") + 1
            name = re.compile(r"\s*(\w+)\s*\(").match(src, at)
            end = _closing(src, name.end() - 1, "()")
            brace = src.index("{", end)
            body = src[brace:_closing(src, brace, "{}")]
            if re.search(r"\bpdl_wait\(|\bmulti_block\(", body):
                out.append((name.group(1), src[name.end():end]))
    return out


def test_early_kernels_do_not_promise_read_only_inputs():
    kernels = early_kernels()
    names = [n for n, _ in kernels]
    for expected in ("stream_collide_kernel", "stream_collide_quad_kernel",
                     "stream_collide_kernel_multi", "face_kernel_multi", "interp_kernel_multi"):
        assert expected in names
    bad = [(n, p.strip()) for n, params in kernels for p in params.split(",")
           if "const" in p and "__restrict__" in p and re.search(r"(\w+)\s*$", p).group(1) not in TABLES]
    assert not bad, bad
