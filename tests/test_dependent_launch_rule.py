"""Kernels launched behind a running one (launch_after) read what it writes with coherent loads.

CUDA defines the non-coherent path (__ldg, and what the compiler may load through a
const __restrict__ kernel parameter) for data that nothing writes while the kernel lives, and such
a kernel lives from before the writes on.  So a kernel that passes wait_for_primary, and every device function
that it reaches, holds no __ldg, and its pointer parameters are not __restrict__ -- but for the tables that the
host had written before the first launch."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_04463_gb300", "csrc")
HOST_TABLES = {"sets", "tile_set", "block_set", "order_sets", "rblock_set", "order", "mblock_set"}


def _functions():
    """name -> [(is a kernel, parameters, body)] of every function of the sources."""
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\b(\w+)\s*\(([^;{}()]*(?:\([^()]*\)[^;{}()]*)*)\)\s*(?:const\s*)?\{", text):
            if m.group(1) in ("if", "for", "while", "switch", "constexpr", "__launch_bounds__"):
                continue
            depth, end = 1, m.end()
            while depth and end < len(text):
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            head = text[max(text.rfind(c, 0, m.start()) for c in ";}{") + 1:m.start()]
            out.setdefault(m.group(1), []).append(("__global__" in head, m.group(2), text[m.end():end]))
    return out


FUNCTIONS = _functions()
WAITING = sorted(n for n, fs in FUNCTIONS.items() for k, _, body in fs if k and "wait_for_primary()" in body)


def test_the_kernels_are_found():
    assert {"k_mirror", "k_count_order", "k_order_table", "k_bucket_scan", "k_action_final", "k_batch_rank",
            "k_batch_action"} <= set(WAITING)
    launched = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        launched |= set(re.findall(r"launch_after\((k_\w+)", open(path).read()))
    assert launched <= set(WAITING)


def test_coherent_loads_after_the_wait():
    wrong = []
    for kernel in WAITING:
        for is_kernel, params, body in FUNCTIONS[kernel]:
            for p in params.split(","):
                if "__restrict__" in p and re.findall(r"\w+", p)[-1] not in HOST_TABLES:
                    wrong.append(f"{kernel}: parameter {p.strip()}")
            seen, todo = set(), [(kernel, body)]
            while todo:
                name, text = todo.pop()
                if "__ldg(" in text:
                    wrong.append(f"{kernel}: __ldg in {name}")
                for callee in set(re.findall(r"\b(\w+)\s*(?:<[^<>;]*>)?\s*\(", text)) | set(re.findall(r"\b([A-Z]\w+)<G> ", text)):
                    if callee in FUNCTIONS and callee not in seen:
                        seen.add(callee)
                        todo += [(callee, b) for k, _, b in FUNCTIONS[callee] if not k]
    assert not sorted(set(wrong)), "\n".join(sorted(set(wrong)))
