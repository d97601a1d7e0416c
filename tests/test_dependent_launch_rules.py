"""The rules of dependent launches (csrc/mh_internal.cuh), read from the sources: a kernel that is launched
by mh_launch_dep waits (mh_dep_wait), and such a kernel reads through the read-only path (const __restrict__
parameters, __ldg) only what is laid out at set-up, never what a kernel before it on the stream writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1007_5335_gb300", "csrc")

# parameters that hold set-up data or a caller's input, by name; kernel-specific ones by "kernel.name"
SETUP = set("""A Al Ah geo curve_of nn off foff coff xy fine tc tr fine32 ccf crad fg tw geo32
    pair_tgt grp_curve grp_pair line_tgt line_curve lag lw woff idx
    img img_off_op kpad_op chunk_op chunk_t0 tc_src task_src task_dst op_of ops op_off op_C perm tab at
    dst_off dst_ptr dst_task chunks out_red row box child region ext_const boxes leaf_box xi bw leaf
    nodes leaf_red flat_idx dxy dnrm leaf_c flat32 bias
    k_dlp_coarse32.src k_cols.src k_loss_dz.t""".split())
NOT_SETUP = {"k_gemm.A"}   # the network's products: activations of the layer before


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__ void[^;{]*?\b(k_\w+)\(([^;{]*?)\)\s*\{", text, re.S):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield m.group(1), m.group(2), text[m.end():end]


def test_dependent_kernels_read_plainly():
    bad, waiting = [], set()
    for name, sig, body in _kernels():
        if "mh_dep_wait()" not in body:
            continue
        waiting.add(name)
        params = [p.strip() for p in sig.split(",")]
        ro = {re.search(r"(\w+)(?:\s*=.*)?$", p).group(1) for p in params if re.search(r"const [^*]*\*\s*__restrict__", p)}
        bad += [f"{name}({p})" for p in ro if f"{name}.{p}" in NOT_SETUP or not (p in SETUP or f"{name}.{p}" in SETUP)]
        if "__ldg" in body:
            bad.append(f"{name}: __ldg")
    assert not bad, bad
    assert len(waiting) > 30


def test_dependent_launches_go_to_kernels_that_wait():
    waiting = {name for name, _, body in _kernels() if "mh_dep_wait()" in body}
    launched = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"mh_launch(?:_dep)?\(([^;]*?)dim3\(", text, re.S):
            launched |= set(re.findall(r"\bk_\w+", m.group(1)))
        launched |= set(re.findall(r"\bkern = (?:gmres_k::)?(k_\w+)", text)) | set(re.findall(r"launch\((k_\w+)", text))
        launched |= set(re.findall(r"launch_cluster\(ctx, gmres_k::(k_\w+)", text))
    assert launched and launched <= waiting, launched - waiting
