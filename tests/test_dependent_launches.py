"""Kernels launched before their predecessor's end (launch_dependent, or the attribute itself) read what it wrote: their sources must
not ask for the non-coherent load path, which is for data that is constant while the kernel lives.  Source check, no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_03260_b200", "csrc")


def functions(text):
    """name -> (parameters, body) of the kernels and device functions"""
    found = {}
    for m in re.finditer(r"__(?:global|device)__[^;{(]*(?:__launch_bounds__\([^{]*?\)\s*)?\b(\w+)\s*\(([^{;]*)\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        found[m.group(1)] = (m.group(2), text[m.end():i])
    return found


def with_callees(name, funcs):
    """[(parameters, body)] of the function and of the functions of these files that it calls"""
    todo, seen = [name], []
    while todo:
        f = todo.pop()
        if f not in seen:
            seen.append(f)
            todo += [c for c in re.findall(r"\b(\w+)\s*(?:<[^;()]*>)?\s*\(", funcs[f][1]) if c in funcs]
    return [funcs[f] for f in seen]


def sources():
    """file -> text without comments, headers of the same folder included"""
    read = lambda f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
    headers = "".join(read(f) for f in sorted(os.listdir(CSRC)) if f.endswith(".cuh"))
    return {f: headers + read(f) for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")}


def test_dependent_kernels_use_plain_loads():
    seen = set()
    for f, text in sources().items():
        funcs = functions(text)
        for name in re.findall(r"__global__[^;{(]*(?:__launch_bounds__\([^{]*?\)\s*)?\b(\w+)\s*\(", text):
            parts = with_callees(name, funcs)
            if not any("dep_wait()" in body for _, body in parts):
                continue
            seen.add(name)
            assert not re.search(r"const[^,]*__restrict__", funcs[name][0]), (f, name)
            # (the bias is older than the fold kernel that precedes the one place where it is read)
            assert not any("__ldg" in body.replace("__ldg(bias + g)", "") for _, body in parts), (f, name)
    assert seen >= {"assign_kernel", "assign_hidden_kernel", "fold_router_kernel", "decode_partial_kernel",
                    "decode_merge_kernel", "summarise_kernel", "group_tiles_kernel", "live_kernel", "focus_attn_kernel"}, seen


def test_every_dependent_launch_waits():
    """a kernel given the attribute must execute the wait"""
    for f, text in sources().items():
        funcs = functions(text)
        for m in re.finditer(r"launch_dependent\(\s*(?:\w+ \? )?(\w+)", text):
            name = m.group(1)
            if name == "kern":
                name = re.findall(r"auto kern = (\w+)", text[:m.start()])[-1]
            if name in funcs:
                assert any("dep_wait()" in body for _, body in with_callees(name, funcs)), (f, name)
            else:
                assert name == "void", (f, name)             # the declaration of launch_dependent itself
