"""Kernels launched over the end of their predecessor (launch_chained) are
resident beside it. Read-only loads (__ldg, pointers both const and
__restrict__) are allowed in them only for arrays that no chained kernel
writes. No run shows a breach reliably, so the sources are read."""
import glob
import os
import re

from paper_2106_15789_gb300 import build

# the cube, the smoothed cube, the masks and the 16-bit cube: written by plain
# launches only, or by the clip, which is over before the next pair begins
READ_ONLY = {"x", "src", "C", "mbits", "m4", "s4", "h16.bits", "h16.scale"}


def _without_comments(text):
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


def _block(text, start, left, right):
    """The text from the first `left` at or after start to its matching `right`."""
    i = j = text.index(left, start)
    depth = 0
    while True:
        depth += (text[j] == left) - (text[j] == right)
        j += 1
        if depth == 0:
            return text[i:j]


def _kernels():
    text = "\n".join(_without_comments(open(p).read()) for p in sorted(glob.glob(os.path.join(build.CSRC, "*.cu"))))
    names = set(re.findall(r"launch_chained\((k_\w+)", text))
    assert len(names) >= 9
    for name in sorted(names):
        at = next(m.end() for m in re.finditer(rf"\b{name}\(", text) if re.search(r"__global__[^;{{}}]*$", text[:m.start()]))
        params = _block(text, at - 1, "(", ")")
        yield name, params, _block(text, at - 1 + len(params), "{", "}")


def test_chained_kernels_read_only_what_none_of_them_writes():
    for name, params, body in _kernels():
        for p in params[1:-1].split(","):
            if re.search(r"\bconst\b", p) and "__restrict__" in p:
                assert p.split()[-1].strip() in READ_ONLY, (name, p)
        for m in re.finditer(r"__ldg\(", body):
            base = re.match(r"\(\s*(?:reinterpret_cast<[^>]*>\()?([\w.]+)", body[m.end() - 1:])
            assert base and base.group(1) in READ_ONLY, (name, body[m.start(): m.end() + 40])


def test_chained_kernels_wait_first():
    """A chained kernel begins with chain_begin() (the counting instance of
    k_share_list, a plain launch, only lets its successor start)."""
    for name, _, body in _kernels():
        head = body[: body.index("chain_begin()")]
        assert not re.search(r"\[[^\]]*\]\s*=[^=]|st->\w|__ld|atomic", head), (name, head)
