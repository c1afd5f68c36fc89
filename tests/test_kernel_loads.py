"""The kernels of a step start as programmatic dependents: a kernel's blocks
may be resident while its predecessors still write the engine's state.  What a
step writes must therefore never go through the read-only path (__ldg), which
promises data that nobody writes in the kernel's life.  Read from the source:
a stale line would show on a GPU only now and then."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRITTEN = {"V", "J", "Ibg", "ref", "acc", "slot_emit", "dyn", "cnt", "bw", "ylast", "closed", "hist", "hcount",
           "hseg", "hr0", "events", "flags"}


def _arguments(text, name):
    """The argument texts of every call of name in text."""
    out = []
    for m in re.finditer(r"\b%s(?:<[\w, ]*>)?\(" % name, text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        out.append(text[m.end():i - 1])
    return out


def test_written_state_is_not_read_through_the_read_only_path():
    src = open(os.path.join(ROOT, "paper_2211_15963_gb300", "csrc", "kernels.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    # per-step delivery is launched plainly: its read-only loads (ld_ring) stay
    a = src.index("__device__ __forceinline__ T ld_ring(")
    b = src.index("constexpr unsigned long long kRowMask")
    body = src[a:b]
    rest = src[:a] + src[b:]
    assert "k_deliver" not in "".join(re.findall(r"launch_after\(([^;]*);", src))
    assert _arguments(body, "ld_ring") and not _arguments(rest, "ld_ring")
    loads = _arguments(rest, "__ldg") + _arguments(rest, "ld_stream_u32") + _arguments(rest, "ld_stream_u64")
    assert len(loads) > 20
    for arg in loads:
        used = set(re.findall(r"\be\.(\w+)", arg))
        assert not used & WRITTEN, arg
