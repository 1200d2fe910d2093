"""Which data the kernels read through the read-only path.  Kernels launched
as programmatic dependents are resident while the kernel ahead still writes, so
what any kernel writes (fields, accumulators, sums) may not be read that way;
what remains are the potential and tables, written before the first launch."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_02891_gb300", "csrc")


def _sources():
    out = {}
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(p, encoding="utf-8").read()
        out[os.path.basename(p)] = re.sub(r"//[^\n]*", "", text)
    return out


def _calls(text, name):
    return [text[m.end():m.end() + 24].strip() for m in re.finditer(rf"\b{name}(?:<[^>]*>)?\(", text)]


def test_read_only_path_is_for_constants():
    src = _sources()
    dependents = {f for f, t in src.items() if "pdl_wait()" in t}
    assert {"ops_impl.cuh", "lines2d.cuh", "lines3.cuh", "fused2d.cuh", "prolong.cuh", "pass_f32.cuh"} <= dependents
    # persist_lines.cuh: a cooperative launch with plain edges, whose X^k and P_k nobody writes meanwhile
    assert "launch_pdl" not in src["persist_lines.cuh"]
    for f, t in src.items():
        raw = _calls(t, "__ldg")
        if f == "ops_impl.cuh":
            assert raw == ["p); }"] or [r[:2] for r in raw] == ["p)"], raw   # ld_const itself
        elif f != "persist_lines.cuh":
            assert not raw, (f, raw)
        for arg in _calls(t, "ld_const"):
            assert re.match(r"const X\*|Vp \+|fine \+", arg), (f, arg)
        assert not re.search(r"ld\.global\.nc|ldv<2>", t), f
        # const __restrict__ parameters of a kernel may be read that way by the compiler: coordinates only
        if f in dependents:
            for k in re.finditer(r"__global__[^{;]*", t):
                for m in re.finditer(r"const[\w\s:<>]+\*\s*__restrict__\s+(\w+)", k.group(0)):
                    assert m.group(1) in ("rx", "ry"), (f, m.group(0))
