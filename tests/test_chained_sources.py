"""Kernels that are launched while their predecessor still runs (chain_enter) read nothing that a
predecessor writes through the read-only path: no __ldg and no const __restrict__ parameter in
them, nor in the functions through which they read fields."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_02652_gb300", "csrc")
# functions by which the chained kernels read fields and intermediate matrices
READERS = {"load_fmunu": "clover.cu", "clink<double>": "clover.cu", "clink<float>": "clover.cu", "load_H": "force.cu",
           "load_d": "force.cu", "load_half_rt": "force.cu", "clover_insert_pair": "force.cu", "hop_force_dir": "force.cu"}


def _block(text, start):
    """The text from start to the end of the brace block that opens after it."""
    i = text.index("{", start)
    depth = 0
    for k in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[start:k + 1]
    raise AssertionError("unbalanced braces")


def _sources():
    return {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read()) for f in glob.glob(os.path.join(CSRC, "*.cu*"))}


def _read_only(block):
    return re.findall(r"__ldg|const[^,(){};]*\*\s*(?:const\s+)?__restrict__\s+\w+", block)


def test_chained_kernels():
    seen = 0
    for name, text in _sources().items():
        for m in re.finditer(r"__global__", text):
            kernel = _block(text, m.start())
            if "chain_enter(" not in kernel:
                continue
            seen += 1
            assert not _read_only(kernel), (name, kernel[:200], _read_only(kernel))
            # load_spinor, load_link18: read-only path unless told otherwise
            assert not re.search(r"\bload_spinor\(|\bload_link18\(", kernel), (name, kernel[:200])
    assert seen >= 20


def test_their_readers():
    src = _sources()
    for fn, name in READERS.items():
        at = [m.start() for m in re.finditer(re.escape(fn) + r"\(", src[name])]
        defs = [b for b in (_block(src[name], i) for i in at if "{" in src[name][i:]) if re.match(re.escape(fn) + r"\([^;{]*\)\s*\{", b)]
        assert defs, fn
        for b in defs:
            assert not _read_only(b), (fn, _read_only(b))
            assert not re.search(r"\bload_spinor\(|\bload_link18\(", b), fn
    # the FP32 spinor loads of the shared-site stencil
    for fn in ("load_spin", "load_comp"):
        b = _block(src["hop_tile.cuh"], src["hop_tile.cuh"].index("> " + fn + "(" if fn == "load_comp" else fn + "("))
        f32 = re.search(r"if constexpr \(PREC == PFMP_F32\) \{(.*?)\} else", b, re.S)
        assert f32 and "__ldg" not in f32.group(1) and "ld_live" in f32.group(1), fn
