"""What the kernel sources have to keep to and no run can show reliably."""
import glob
import os
import re

from paper_2403_16122_gb300 import build as lbm_build


def _code(name):
    """Source text without comments."""
    txt = open(os.path.join(lbm_build.CSRC, name)).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", txt), flags=re.S)


def _body(src, name):
    """The body of the function `name` (its last definition)."""
    at = [m.start() for m in re.finditer(r"\b%s\(" % name, src)]
    for start in reversed(at):
        brace = src.find("{", start)
        semi = src.find(";", start)
        if brace < 0 or (0 <= semi < brace):
            continue
        depth = 0
        for k in range(brace, len(src)):
            depth += {"{": 1, "}": -1}.get(src[k], 0)
            if depth == 0:
                return src[brace:k + 1]
    raise AssertionError(name)


def test_no_read_only_loads_of_data_still_being_written():
    """A kernel that is resident before the grid ahead of it has ended (launched
    as a programmatic dependent) or that reads what other CTAs stored during its
    own run (persistent) must not read that data on the read-only path, nor
    through intrinsics that the compiler may move ahead of the wait. The
    read-only path is left to the strips that load in place, launched after the
    grid before them has ended."""
    srcs = {os.path.basename(p): _code(os.path.basename(p))
            for p in glob.glob(os.path.join(lbm_build.CSRC, "*.cu*"))}
    for name, src in srcs.items():
        assert "__ldcg" not in src and "ld.global.nc" not in src, name
        want = 1 if name == "lbm_kernels.cu" else 0  # ld_state, read-only path
        assert src.count("__ldg(") == want, name
    kern, block, red = srcs["lbm_kernels.cu"], srcs["lbm_block.cuh"], srcs["lbm_reduce.cu"]
    # which path each kernel body takes
    item = _body(kern, "strip_item")
    assert "kPath = PERSIST ? Path::kL2 : (STG == 0 ? Path::kReadOnly : Path::kOrdered)" in item
    assert kern.count("Path::kReadOnly") == 2  # there and in ld_state
    persist = {k: re.findall(r"strip_item<\w+, \w+, (\w+)", _body(kern, k))
               for k in ("step_strip", "step_strip_staged", "step_strip_noalloc",
                         "step_strip_persistent")}
    assert persist == {"step_strip": ["false"], "step_strip_staged": ["false"],
                       "step_strip_noalloc": ["false"], "step_strip_persistent": ["true"]}
    assert "block_item<OBS, ST, Path::kOrdered>" in _body(kern, "step_block")
    assert "block_item<false, ST, Path::kL2>" in _body(kern, "step_block_persistent")
    assert "kReadOnly" not in block
    # strips that load in place: a plain launch, no dependent start
    in_place = _body(kern, "launch_strip_w")
    assert "<<<" in in_place and "ProgrammaticStreamSerialization" not in in_place
    # the reductions' partials come as const __restrict__ parameters: ld_live only
    assert re.findall(r"\brow\s*[\[+][^;]*", _body(kern, "reduce_noalloc")) == \
        ["row + p0 + 32 * k) : 0.0"]
    assert "ld_live(row + p0 + 32 * k)" in kern
    assert "ld_live(p + (c + 8 * k) * stride)" in _body(red, "sum_values")


def test_whole_file_compilation_defines_every_entry():
    """lbm_kernels.cu compiled without LBM_PART holds every part: each function
    that lbm_internal.h declares is defined by it or by another source."""
    import subprocess

    cmd = [lbm_build.nvcc(), *lbm_build.ARCH, "-std=c++17", f"-I{lbm_build.INCLUDE}",
           f"-I{lbm_build.CSRC}", "-E", os.path.join(lbm_build.CSRC, "lbm_kernels.cu")]
    txt = subprocess.run(cmd, capture_output=True, text=True, check=True).stdout
    txt += _code("lbm_api.cu")
    header = _code("lbm_internal.h")
    names = re.findall(r"^(?:cudaError_t|int|bool|void) (\w+)\([^{};]*\);", header, flags=re.M)
    assert len(names) >= 20 and "launch_step_noalloc_strip" in names
    missing = [n for n in names if not re.search(r"\b%s\([^{};]*\)\s*\{" % n, txt)]
    assert missing == []


def test_state_transfer_waits_for_its_copies_after_a_failure_too():
    """lbm_get_state and lbm_set_state in FP32 storage copy plane by plane between
    the device and the caller's arrays, which may be pinned: copies queued before
    a call that fails still run. The stream is waited for on every way out."""
    api = _code("lbm_api.cu")
    for name in ("get_state_fp32", "set_state_fp32"):
        body = _body(api, name)
        wait = body.index("cudaStreamSynchronize")
        # unconditional, and no way out of the function before it
        assert re.search(r"\n    const cudaError_t \w+ = cudaStreamSynchronize", body), name
        outer = re.sub(r"auto (planes|plane) = \[&\].*?\n    \};|auto plane = [^;]*;[^;]*;",
                       "", body[:wait], flags=re.S)
        assert "return" not in outer, name
