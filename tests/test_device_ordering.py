"""Ordering rules of the device code that no run can show to be kept, checked
on the source (csrc/): a kernel that lets its successor start early
(dep_release, common.cuh) allocates its tensor memory first."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2504_14494_gb300", "csrc")
ALLOC = re.compile(r"\b(tc_setup|tc_setup_groups|tmem_alloc)\(")
RELEASE = re.compile(r"(?<!return )\bdep_(sync|release)\(\)")  # `return dep_sync()`: the CTA ends


def _strip(src):
    src = re.sub(r"/\*.*?\*/", lambda m: re.sub(r"[^\n]", " ", m.group()), src, flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _close(src, i, pair):
    depth = 0
    for j in range(i, len(src)):
        depth += {pair[0]: 1, pair[1]: -1}.get(src[j], 0)
        if depth == 0:
            return j
    raise AssertionError("unbalanced " + pair)


def functions():
    """{name: (parameters, body)} of the kernels and device functions of csrc/."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = _strip(open(path).read())
        for m in re.finditer(r"__(?:global|device)__", src):
            i = m.end()
            head = re.compile(r"\b(\w+)\s*\(").search(src, i)
            while head and head.group(1) in ("__launch_bounds__", "__noinline__"):
                head = re.compile(r"\b(\w+)\s*\(").search(src, _close(src, head.end() - 1, "()") + 1)
            if not head:
                continue
            end = _close(src, head.end() - 1, "()")
            rest = re.compile(r"\s*(const)?\s*\{").match(src, end + 1)
            if rest:
                out[head.group(1)] = (src[head.end():end],
                                      src[rest.end() - 1:_close(src, rest.end() - 1, "{}") + 1])
    return out


def test_tensor_memory_is_allocated_before_the_successor_is_released():
    seen = set()
    for name, (_, body) in functions().items():
        release = RELEASE.search(body)
        allocs = list(ALLOC.finditer(body))
        callee = re.search(r"\bmlp_or_encode\b|\bmlp_only_step\b", body)
        if release and (allocs or callee):
            last = max([a.start() for a in allocs] + ([callee.start()] if callee else []))
            assert last < release.start(), f"{name} releases its successor before it allocates"
            seen.add(name)
    # every kernel of the early-launched calls that uses tensor memory
    assert {"gnn_encode_kernel", "gnn_round_kernel", "gnn_head_bwd_kernel", "gnn_round_bwd1_kernel",
            "gnn_round_bwd2_kernel", "gnn_encode_bwd_kernel", "mlp_or_encode"} <= seen
