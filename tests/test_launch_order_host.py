"""Kernels launched behind the previous one (launch_behind) are resident while it
still writes.  What keeps their reads behind its end is behind_previous(), and that
holds only where the compiler may not move a load across it or take the
non-coherent path (which wants data that nothing writes during the kernel's whole
life).  Both are granted by a `__restrict__` pointer and by `__ldg`, so the sources
of such kernels, and of the device functions they call, hold neither."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2603_09277_gb300", "csrc")
# launched by itself (cooperative, or as one cluster): starts after the previous
# kernel has ended, its inputs are written by none of its own blocks
PLAIN = {"depth_sort_kernel"}


def _code():
    """{file: source without comments}"""
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        s = re.sub(r"/\*.*?\*/", " ", open(f).read(), flags=re.S)
        out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", s)
    return out


def _close(s, i, a, b):
    """The index behind the bracket that closes the one at s[i]."""
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == a) - (s[j] == b)
        if depth == 0:
            return j + 1
    raise AssertionError("unbalanced")


def _kernels(s):
    """(name, start, end of the parameters, body) of every kernel definition of s"""
    for m in re.finditer(r"__global__\s+void\s+", s):
        at = m.end()
        if s.startswith("__launch_bounds__", at):
            at = _close(s, s.index("(", at), "(", ")")
        n = re.compile(r"\s*(\w+)\s*\(").match(s, at)
        args = _close(s, n.end() - 1, "(", ")")
        if not re.compile(r"\s*\{").match(s, args):
            continue  # a declaration
        body = s.index("{", args)
        yield n.group(1), m.start(), args, s[body + 1:_close(s, body, "{", "}") - 1]


def test_kernels_wait_first_and_read_through_coherent_loads():
    code = _code()
    kernels, behind = {}, set()
    for f, s in code.items():
        for name, start, args, body in _kernels(s):
            kernels[name] = body
            if name in PLAIN:  # (its own text is not held to the rule)
                s = s.replace(body, " ")
        behind |= set(re.findall(r"launch_behind\(\s*(\w+)", code[f]))
        for banned in ("__restrict__", "__ldg", "ld.global.nc", "__builtin_nontemporal_load"):
            assert banned not in s, "%s holds %s" % (f, banned)
    behind.discard("void")  # (the definition)
    assert len(behind) >= 15 and not behind & PLAIN
    for name in behind:
        assert re.match(r"\s*behind_previous\(\);", kernels[name]), name
    assert set(kernels) - behind == PLAIN
