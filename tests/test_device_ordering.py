"""Ordering rules of the device code that no run can show to be kept, checked
on the source (csrc/): a kernel that lets its successor start early
(dep_release, common.cuh) allocates its tensor memory first, and a kernel that
starts early reads its predecessor's outputs by loads that stay where they are
(ld_prev); a wait for what another CTA of a cluster sends acquires at cluster
scope."""
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


# Buffers that the kernel before may still be writing when a kernel launched
# early starts (None: it may be the first kernel of a call, so all of them).
PREVIOUS = {
    "gnn_pack_kernel": None, "adamw_kernel": None, "gnn_head_bwd_kernel": None,
    "gnn_collide_loss_kernel": None,
    "gnn_round_kernel": ["h_src", "ra.ab_in"],      # the encoder's or the round's before
    "loss_finish_kernel": ["lossp"],
    "gnn_collide_adjoint_kernel": ["g_in"],         # stream_adjoint_sum_kernel's
    "stream_adjoint_sum_kernel": [],                # follows grad_reduce_kernel, reads older outputs
    "gnn_round_bwd1_kernel": ["dh_out"],            # the head's or the edge backward's
    "gnn_round_bwd2_kernel": ["da", "dh_part"],
    "gnn_encode_bwd_kernel": ["dh0"],
    "grad_reduce_kernel": ["G"],
}
LOADERS = ("ld_pf", "ld_pf32", "copy_row", "blob_ok")


def test_outputs_of_the_kernel_before_are_not_declared_unchanged():
    """What the kernel before an early-launched one writes is read at addresses
    formed after the wait, without __ldg and without a const __restrict__
    pointer (both promise that the data does not change while the kernel
    runs)."""
    funcs = functions()
    for name in LOADERS:
        assert "__ldg(" not in funcs[name][1], name
    early = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = _strip(open(path).read())
        early |= set(re.findall(r"launch_after\(\s*[^,()]*(?:==[^,()]*)?,\s*(?:kern\b|(\w+))", src))
    # (those launched through `kern`, by the size of the call)
    early = {n for n in early if n} | {"gnn_round_bwd1_kernel", "gnn_round_bwd2_kernel",
                                       "gnn_encode_bwd_kernel"}
    assert early == set(PREVIOUS)
    pointer = re.compile(r"const\s+\w+\s*\*\s*(__restrict__\s+)?(\w+)")
    for name, buffers in PREVIOUS.items():
        params, body = funcs[name]
        if buffers is None:
            assert "__ldg(" not in body and "copy_g2s(" not in body, name
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params), name
            buffers = [m.group(2) for m in pointer.finditer(params)]
        for b in buffers:
            assert not re.search(r"__ldg\((?:chunk[48]\()?" + re.escape(b) + r"\b", body), (name, b)
            assert b not in [m.group(2) for m in pointer.finditer(params) if m.group(1)], (name, b)
        if buffers:
            wait = max(m.end() for m in re.finditer(r"(?<!return )\bdep_(?:sync|wait)\(\)", body))
            taken = [m.start() for m in re.finditer(r"\bafter_wait\(", body)]
            assert taken and min(taken) > wait, name


def test_waits_for_another_cta_acquire_at_cluster_scope():
    senders = 0
    for name, (_, body) in functions().items():
        if re.search(r"\bst_async\(", body) and name != "st_async":
            senders += 1
            assert not re.search(r"\bmbar_(?:try_)?wait(?:_sleep)?(?:<false>)?\(", body), name
            assert "mbar_wait<true>(" in body, name
    assert senders == 1  # the resident multi-step kernel
    body = functions()["mbar_try_wait_sleep"][1]
    assert "try_wait.parity.acquire.cluster." in body[:body.index("else")]


def test_collisions_spell_out_their_roundings():
    """A product and a sum written with operators may or may not be contracted,
    kernel by kernel; the BGK collision, which single-step and multi-step calls
    share (equal bit for bit), uses none."""
    funcs = functions()
    for name in ("rho9", "mom9", "usq9", "feq_poly", "bgk_relax", "bgk_collide", "bgk_collide_fast",
                 "bgk_collide_pair"):
        body = funcs[name][1].replace("3.0f * sign", "")  # (exact: sign is +-1)
        assert not re.search(r"[\w)\]] [*+-] [\w(]|[*+-]=", body), name
    src = "".join(_strip(open(p).read()) for p in glob.glob(os.path.join(CSRC, "*.cu*")))
    assert len(re.findall(r"void bgk_collide\(", src)) == 1
    for kernel in ("bgk_step_x4", "bgk_step_any", "bgk_batch_kernel", "pair_residual_kernel"):
        assert "bgk_collide(" in funcs[kernel][1], kernel
