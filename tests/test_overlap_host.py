"""Kernels that may start before the step they continue from has ended
(lbm_pdl.cuh) read what a step writes by plain loads: such data is not
read-only while they run, so neither __ldg nor const __restrict__ pointers
may serve it. Read from the sources; no GPU needed."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_01975_gb300", "csrc")
# never written by a step: solid nodes, a batch's descriptors and items
STEADY = {"mask", "members", "items"}


def sources():
    out = {}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            out[name] = re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)
    return out


def block(text, start):
    """The brace-matched block that begins at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def functions(text, keyword):
    """(name, parameters, body) of every definition with `keyword` before it."""
    for m in re.finditer(keyword + r"[^;{}]*?(\w+)\s*\(", text):
        if m.group(1) == "__launch_bounds__":
            m = re.compile(r"__launch_bounds__\s*\([^{;]*?\)\s*\n\s*(\w+)\s*\(").search(text, m.start())
        depth, j = 1, m.end()
        while depth:
            depth += (text[j] == "(") - (text[j] == ")")
            j += 1
        yield m.group(1), text[m.end():j - 1], block(text, j)


def read_only_params(params):
    return {m.group(1) for m in re.finditer(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params)}


def test_overlapped_kernels_read_by_plain_loads():
    overlapped = {}
    for name, text in sources().items():
        for kernel, params, body in functions(text, "__global__"):
            if "step_wait()" in body:
                overlapped[kernel] = params
    assert {"k_step2d", "k_step2d_batch", "k_force_sweep2", "k_macro", "k_step_f32_wstma",
            "k_step_f32_wstma_batch"} <= set(overlapped), sorted(overlapped)
    bad = {k: read_only_params(p) - STEADY for k, p in overlapped.items() if read_only_params(p) - STEADY}
    assert not bad, bad


def test_their_device_functions_read_by_plain_loads():
    text = sources()
    want = {"tile2d": "lbm_step2d.cuh", "fused_tile_wstma": "lbm_fused_f32_body.cuh",
            "fixed_pops": "lbm_fixed.cuh"}
    for fn, name in want.items():
        found = [p for f, p, _ in functions(text[name], "__device__") if f == fn]
        assert found, fn
        for params in found:
            # (the densities of the TMA-staged shifted form, which is not overlapped)
            assert not read_only_params(params) - STEADY - ({"rho_src"} if fn == "fused_tile_wstma" else set()), fn
    assert "__ldg" not in text["lbm_step2d.cuh"]
    # phase A of the TMA-staged forms (BOXED): nodes that lie in no box
    a = [(p, b) for f, p, b in functions(text["lbm_fused_f32_body.cuh"], "__device__") if f == "phase_a"]
    assert len(a) == 1 and "f" not in read_only_params(a[0][0])
    reads = re.findall(r"[^;]*__ldg\((?!mask)[^;]*;", a[0][1])
    assert len(reads) == 1 and "BOXED ? *q : __ldg(q)" in reads[0], reads
    assert "__ldg" not in next(b for f, _, b in functions(text["lbm_fused_f32_body.cuh"], "__device__")
                               if f == "load_from_box")


def test_only_waiting_kernels_are_launched_overlapped():
    """Every launch that may overlap is of a kernel that waits."""
    text = sources()
    waits = {k for t in text.values() for k, _, b in functions(t, "__global__") if "step_wait()" in b}
    for name, t in text.items():
        if name == "lbm_pdl.cuh":
            continue
        for m in re.finditer(r"lbmpdl::launch_step\(([^,]+),\s*(?:\w+::)*(\w+)", t):
            assert m.group(2) in waits, (name, m.group(2))


def test_room_is_asked_of_the_kernel():
    """Whether a D2Q9 step leaves its successor room follows from the blocks that
    an SM holds of that kernel, not from a number in the source."""
    api = sources()["lbm_api.cu"]
    assert "cudaOccupancyMaxActiveBlocksPerMultiprocessor" in api
    for fn in ("launch_2d_r", "launch_batch_2d_r"):
        body = block(api, api.index("void %s(" % fn))
        assert "leaves_no_room(lbmf2::k_step2d" in body and not re.search(r"\d\s*\*\s*[\w>\[\].-]*sms", body), body
