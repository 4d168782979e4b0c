"""Kernels launched before their predecessor's end (launch_dependent, or the attribute itself) read what it wrote: their sources must
not ask for the non-coherent load path, which is for data that is constant while the kernel lives.  Source check, no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_03260_b200", "csrc")


def kernels(text):
    """name -> (parameters, body) of the __global__ functions"""
    found = {}
    for m in re.finditer(r"__global__[^;{(]*(?:__launch_bounds__\([^{]*?\)\s*)?\b(\w+)\s*\(([^{;]*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        found[m.group(1)] = (m.group(2), text[m.end():i])
    return found


def test_dependent_kernels_use_plain_loads():
    seen = set()
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for name, (params, body) in kernels(text).items():
            if "dep_wait()" not in body:
                continue
            seen.add(name)
            assert not re.search(r"const[^,]*__restrict__", params), (f, name)
            assert "__ldg" not in body, (f, name)
    # and the device functions of the attention kernel
    shared = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "attn_common.cuh")).read() + open(os.path.join(CSRC, "attn_sm100.cu")).read())
    assert "__ldg" not in shared
    assert seen >= {"assign_kernel", "assign_few_kernel", "assign_hidden_kernel", "fold_router_kernel", "decode_partial_kernel",
                    "decode_merge_kernel", "summarise_kernel", "live_kernel", "focus_attn_kernel"}, seen


def test_every_dependent_launch_waits():
    """a kernel given the attribute must execute the wait"""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        ks = kernels(text)
        for m in re.finditer(r"launch_dependent\(\s*(\w+)", text):
            name = m.group(1)
            if name == "kern":
                name = re.findall(r"auto kern = (\w+)", text[:m.start()])[-1]
            assert "dep_wait()" in ks[name][1], (f, name)
