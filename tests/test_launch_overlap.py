"""Kernels that are resident while their predecessor still writes (programmatic dependent launch): nothing in their
source may let the compiler treat what they read as read-only memory.  Read from the source; nothing runs."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_14838_b200", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


def _functions(text):
    """(name, parameters, body) of every kernel and device function."""
    for m in re.finditer(r"__(?:global|device)__[^;{}]*?(\w+)\s*\((?=[^)]*\))", text):
        if m.group(1) == "__launch_bounds__":
            m = re.compile(r"(\w+)\s*\(").search(text, text.index(")", m.end()) + 1)
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, start = text[m.end():i - 1], text.find("{", i)
        depth, j = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield m.group(1), params, text[start:j]


HEADERS = sorted(f for f in os.listdir(CSRC) if f.endswith(".cuh"))


def test_every_kernel_launched_with_overlap_waits():
    launched = set(re.findall(r"launch_pdl\((?:parts > 1 \? )?(\w+)", _source("dkv.cu"))) - {"void"}
    assert {"rb_locate_kernel", "select_gather_cluster_kernel", "shrink_kernel", "decode_split_kernel"} <= launched
    kernels = {n: body for f in HEADERS for n, _, body in _functions(_source(f))}
    for name in launched - {"score_kernel"} | {"score_tc_kernel", "select_topk_kernel", "select_gather_kernel"}:
        assert "pdl_wait();" in kernels[name], name


@pytest.mark.parametrize("header", HEADERS)
def test_no_read_of_such_a_kernel_is_marked_read_only(header):
    text = _source(header)
    assert not re.search(r"__ldg\s*\(|ld\.global\.(?:\w+\.)*nc|__ld(?:lu|cv)\s*\(", text)
    functions = list(_functions(text))
    waiting = [n for n, _, body in functions if "pdl_wait();" in body]
    called = {n for n, _, _ in functions if any(re.search(rf"\b{n}\b", b) for m, _, b in functions if m in waiting)}
    for name, params, _ in functions:
        if name in waiting or name in called or not name.endswith("_kernel"):
            assert "__restrict__" not in params, name


def test_a_warpgroup_changes_its_registers_by_one_instruction():
    """setmaxnreg has to be the same instruction for all warps of a warpgroup, and a block's shares no more than it was launched with."""
    text = _source("score_sweep.cuh")
    kernel = {n: body for n, _, body in _functions(text)}["score_sweep_kernel"]
    changes = re.findall(r"if \(warp (<|>=) kSoftWarps\) \{?\s*asm volatile\(\"setmaxnreg\.(inc|dec)\.", kernel)
    assert sorted(changes) == [("<", "inc"), (">=", "dec")] and text.count("setmaxnreg") == 2
    value = {n: int(v) for n, v in re.findall(r"\b(k\w+) = (\d+)\b", text)}
    soft, warps = value["kSoftWarps"], value["kWarps"]
    assert soft % 4 == 0 and warps % 4 == 0
    at_launch = 65536 // (warps * 32) // 8 * 8
    assert soft * value["kSoftRegs"] + (warps - soft) * value["kOtherRegs"] <= warps * at_launch


def test_kernels_that_early_readers_count_on_start_them_after_their_own_wait():
    """What kernels before the predecessor wrote is complete before a kernel's own wait only if the predecessor has waited itself
    before it lets its successor start."""
    kernels = {n: body for f in HEADERS for n, _, body in _functions(_source(f))}

    def order(body):
        return re.findall(r"\b(pdl_wait|pdl_launch)\(\);", body)

    for name in ("rb_locate_kernel", "rb_collect_kernel", "rb_finish_kernel"):
        assert order(kernels[name]) == ["pdl_wait", "pdl_launch"], name
        head = kernels[name][:kernels[name].index("pdl_launch();")]
        assert head.count("{") - head.count("}") == 1, f"{name}: the order holds for every thread"
    sweep = kernels["score_sweep_kernel"]
    key_sums = sweep.index("if (kSweep == kKeySums) {")
    row_sums = sweep.index("} else {", key_sums)
    assert order(sweep[row_sums:sweep.index("}", row_sums + 1)]) == ["pdl_wait", "pdl_launch"]
    assert order(sweep[:key_sums]) == []
    source = _source("dkv.cu")

    def launches(function):
        body = source[source.index(f"int {function}("):]
        return re.findall(r"\b(rb_\w+_kernel|select_gather\w*_kernel|pool_kernel|score_kernel)\b", body[:body.index("\n}")])

    # the early readers' predecessors are these
    assert launches("do_rebudget") == ["rb_locate_kernel", "rb_collect_kernel", "rb_finish_kernel"]
    assert launches("launch_sweeps").count("pool_kernel") == 1
    body = source[source.index("int do_pass("):]
    assert re.search(r"do_rebudget\(.*\n\s*if \(\(rc = do_select_gather\(", body[:body.index("\n}")])


def test_the_scoring_kernel_of_passes_is_launched_with_overlap_and_waits():
    body = _source("dkv.cu")
    assert re.search(r"auto launch = \[&\]\(auto score_kernel, int smem\) \{ return launch_pdl\(score_kernel,", body)
    kernels = {n: b for n, _, b in _functions(_source("score_sweep.cuh"))}
    assert kernels["score_sweep_kernel"].count("pdl_wait();") >= 4 and "pdl_wait();" in kernels["pool_kernel"]
