"""Which loads may take the read-only path (ld.global.nc), read off the kernel
sources: its contract is that no thread writes the data while the kernel runs.

The persistent launch reads what other blocks of the same launch wrote, so its strip
updates must be instantiated without that path; a per-step kernel is launched as a
dependent of the step before, so it must wait before anything else, and must not let
its own dependents start while its blocks still write."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_00530_gb300", "csrc")


def _source(name):
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", s, flags=re.S)


def _body(src, signature):
    """The braces that follow the first match of `signature`."""
    i = src.index("{", re.search(signature, src).end())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
    return src[i:j]


def test_read_only_loads_stand_in_named_helpers():
    """Step kernels load populations with load_word<RO>; the other two helpers serve
    kernels that are not dependent launches and read what earlier launches wrote."""
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        for helper in (r"load_word\(", r"load_raw\(", r"get_dense\("):
            if re.search(r"__forceinline__ [^;{]*" + helper + r"[^;{]*\)\s*{", src):
                src = src.replace(_body(src, r"__forceinline__ [^;{]*" + helper), "")
        assert "__ldg" not in src and ".nc." not in src, name
    assert "if constexpr (RO) return __ldg(p)" in re.sub(r"\s+", " ", _source("lbm_device.cuh"))


def test_persistent_strips_take_ordinary_loads():
    for name in ("lbm_step_persistent.cuh", "lbm_step_q7.cuh"):
        src = _source(name)
        run = _body(src, r"struct PersistStrip<[79]>")
        assert re.search(r"direct_strip(_q7)?<MODEL, ST, VEC, false, NOISE, false, false>\(", run), name
        assert "load_raw" not in run
    for name, strip in (("lbm_step.cuh", "direct_strip"), ("lbm_step_q7.cuh", "direct_strip_q7")):
        src = _source(name)
        assert re.search(r"bool RAGGED, bool RO(?:, typename Time)?>\s*__device__ __forceinline__ void " + strip + r"\(", src)
        # every population load of the strip names its path
        assert not re.search(r"load_vec<ST, VEC>\(", src)


def test_per_step_kernels_wait_before_populations_and_release_after_them():
    for name, kernel, strip, stores in (("lbm_step.cuh", "step_kernel", "direct_strip", "store_vec<"),
                                        ("lbm_step_q7.cuh", "step_kernel_q7", "direct_strip_q7", "q7_row<")):
        src = _source(name)
        body = _body(src, r"\b" + kernel + r"\(const StepArgs a\)")
        # the wait comes first, or in time(), which the strip calls before it reads a buffer's address
        call = body[body.index(strip + "<"):]
        first = body[1:].lstrip().startswith("wait_for_previous();")
        either = re.search(r"if constexpr \(!(\w+)\) wait_for_previous\(\);", body[:body.index(strip + "<")])
        late = bool(either) and f"if constexpr ({either[1]}) wait_for_previous();" in call[:call.index("});")]
        assert first or late, name
        assert "allow_dependents" not in body
        update = _body(src, r"__forceinline__ void " + strip + r"\(")
        assert update.index("time()") < update.index("dp->f[")
        # dependents only after the stores of the strip's last row
        assert update.count("allow_dependents") == 1
        release = update.index("allow_dependents")
        assert release > update.rindex(stores)
        assert re.search(r"y \+ [12] (==|>=) y_end\) $", update[:release]), name
