"""Kernels started by launch_chain may begin while their predecessor still runs, so nothing of them may read memory
before chain_begin()'s wait.  Checked in the source (no GPU needed):

- every kernel handed to launch_chain begins with chain_begin();
- none of its parameters is __restrict__: loads through const __restrict__ pointers count as invariant over the whole
  kernel, and a load that cannot change may be moved above the wait.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0811_4331_gb300", "csrc")


def _sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        out[os.path.basename(path)] = re.sub(r"\\\n", "\n", src)
    return out


def _balanced(src, i, opening, closing):
    depth = 0
    for k in range(i, len(src)):
        depth += (src[k] == opening) - (src[k] == closing)
        if depth == 0:
            return k
    raise AssertionError("unbalanced source")


def _kernels(src):
    """name -> (parameter list, first statement of the body)"""
    out = {}
    for m in re.finditer(r"__global__\s+void\s+", src):
        i = m.end()
        if src.startswith("__launch_bounds__", i):
            i = _balanced(src, src.index("(", i), "(", ")") + 1
        name = re.match(r"\s*(\w+)\s*\(", src[i:])
        p0 = i + name.end() - 1
        p1 = _balanced(src, p0, "(", ")")
        body = re.match(r"\s*\{\s*([^;]*;)", src[p1 + 1:])
        if body:
            out[name.group(1)] = (src[p0:p1 + 1], body.group(1))
    return out


def _chained(src):
    """Names of the kernels that launch_chain is given: directly, through `auto k = kernel<...>`, or through a
    function whose body names the kernels it chooses from."""
    names = set()
    for m in re.finditer(r"launch_chain\(\s*(\w+)", src):
        back = re.findall(r"auto\s+%s\s*=\s*(\w+)\s*[<;]" % m.group(1), src[:m.start()])
        name = back[-1] if back else m.group(1)
        if name.endswith("_kernel"):
            names.add(name)
            continue
        f = re.search(r"\b%s\([^)]*\)[^{;]*\{" % name, src)
        assert f, name
        inner = set(re.findall(r"\b(\w+_kernel)\b", src[f.end():_balanced(src, f.end() - 1, "{", "}")]))
        assert inner, name
        names |= inner
    return names


def test_chained_kernels_wait_first_and_hold_no_restrict_pointers():
    seen = 0
    for name, src in _sources().items():
        kernels = _kernels(src)
        for k in _chained(src):
            assert k in kernels, (name, k)
            params, first = kernels[k]
            assert first == "chain_begin();", (name, k, first)
            assert "__restrict__" not in params, (name, k)
            seen += 1
    assert seen >= 30
