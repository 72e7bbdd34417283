"""Kernels launched programmatically live while their predecessors in the stream still write.  Read off the sources, no GPU: nothing but
weight tiles (TMA) is loaded before a kernel's dependency wait, and nothing is loaded through the non-coherent path, which takes
memory to be read-only for the kernel's lifetime.  (A wrong value from such a load is a matter of timing, so running the kernels shows
it only now and then.)"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_23367_b200", "csrc")
ORDINARY = {"restore_kept_cluster_kernel"}     # launched as ordinary stream work: its predecessors are complete
LOADS = r"\b(?:dep_load\w*|x_load\w*|load16|load_row8|load_index|load4_any|stage_bias|__ldg|__ldcg|__ldcs)\s*\("


def _strip(text):
    return re.sub(r"//[^\n]*", "", text)


def _kernels():
    """(file, name, parameter list, body) of every __global__ function."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _strip(open(path).read())
        for m in re.finditer(r"__global__\b", text):
            head = re.compile(r"(\w+)\s*\(").finditer(text, m.end())
            name = next(h for h in head if h.group(1) not in ("__launch_bounds__",))
            i = name.end()
            depth = 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params = text[name.end():i - 1]
            j = text.index("{", i)
            k, depth = j + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            out.append((os.path.basename(path), name.group(1), params, text[j + 1:k - 1]))
    return out


KERNELS = _kernels()


def _before_the_wait(body):
    """The statements in front of the first wait.  Local functions are taken out (they count where they are called), and one that loads may
    be called there under `early` alone, the launcher's word that nothing still running writes what it reads."""
    head = body[:body.index("pdl_wait()")]
    for m in reversed(list(re.finditer(r"auto (\w+) = \[&\][^{]*\{", head))):
        k, depth = m.end(), 1
        while depth:
            depth += {"{": 1, "}": -1}.get(head[k], 0)
            k += 1
        loads = re.search(LOADS, head[m.end():k])
        head = head[:m.start()] + head[k:]
        if loads:
            for call in re.finditer(r"\b" + m.group(1) + r"\(", head):
                line = head[head.rfind("\n", 0, call.start()) + 1:call.start()]
                assert re.search(r"&& (a\.)?early\)", line), f"{m.group(1)} is called before the dependency wait"
    return head


def test_the_kernels_are_found():
    names = {k[1] for k in KERNELS}
    assert {"gather_ln_kernel", "select_small_kernel", "next_input_kernel", "gemm_cluster_kernel", "restore_bf16_kernel", "score_topk_kernel"} <= names
    assert ORDINARY <= names


@pytest.mark.parametrize("file,name,params,body", KERNELS, ids=[k[1] for k in KERNELS])
def test_loads_of_a_programmatic_kernel(file, name, params, body):
    if "pdl_wait()" not in body:
        assert "pdl_trigger()" not in body
        return
    if name in ORDINARY:
        launches = _strip(open(os.path.join(CSRC, file)).read())
        assert not re.search(r"launch_pdl\(\s*" + name, launches)
        return
    assert not re.search(LOADS, _before_the_wait(body)), "loaded before the dependency wait"
    for chunk in re.split(r"\belse\b", body):           # the GEMM kernels' warp roles wait for themselves
        if "stage_bias(" in chunk and "gemm" in file:
            assert "pdl_wait()" in chunk[:chunk.index("stage_bias(")], "bias staged before the dependency wait"
    assert "__ldg" not in body
    assert not re.search(r"\bconst\s+\w+\s*\*\s*__restrict__", params), "read-only parameters may be loaded non-coherently"


def test_only_a_step_out_of_place_lets_a_launch_read_early():
    api = _strip(open(os.path.join(CSRC, "api.cu")).read())
    calls = re.findall(r"launch_gather_ln\((.*?)\);", api, flags=re.S)
    assert [c.split(",")[-1].strip() == "copied" for c in calls].count(True) == 1
    assert re.search(r"const bool copied = out_dev != tokens_dev && !\(pruned && c\.granularity == 1\);", api)
    assert re.search(r"if \(copied &&\s*cudaMemcpyAsync\(out_dev, tokens_dev", api)


def test_no_other_code_loads_non_coherently():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))):
        text = _strip(open(path).read())
        for file, name, _, body in KERNELS:
            if name in ORDINARY and file == os.path.basename(path):
                text = text.replace(body, "")
        assert "__ldg" not in text, os.path.basename(path)
