"""Kernels that may start while the launch before them drains (pdl.cuh) read
populations that change during their lifetime, so none of those loads may take
the read-only path.  Read from the sources: the read-only path appears only in
LoadReadOnly, which only the batched kernels take, and those are launched in
plain stream order; and for their block records."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1107_4543_gb300", "csrc")
# everything reached by launch_pdl
REACHED = ["d2q9_pull.cuh", "step_impl.cuh", "step_multi.cuh", "step_f64.cu", "step_f32.cu",
           "step_f16.cu", "step_bf16.cu", "step_f64dev.cu", "collide.cuh", "pdl.cuh"]
RECORDS = re.compile(r"__ldg\(reinterpret_cast<const uint32_t \*>\(blocks \+ n?b\) \+ lane\)")
POLICY = re.compile(r"struct LoadReadOnly \{.*?\n\};", re.S)


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def functions(src):
    """(name of the last function or kernel opened before it, use) of each
    step_task call."""
    out = []
    for m in re.finditer(r"step_task<T, (\w+)>\(", src):
        heads = re.findall(r"\b(k_\w+|batch_block)\(const", src[:m.start()])
        out.append((heads[-1], m.group(1)))
    return out


def test_the_read_only_path_is_left_to_kernels_in_stream_order():
    for name in REACHED:
        assert "__ldg" not in RECORDS.sub("", POLICY.sub("", code(name))), name
    uses = functions(code("step_impl.cuh"))
    assert {"k_step_dev", "batch_block", "k_step_batch_stride"} == {k for k, _ in uses}
    for kernel, policy in uses:
        assert policy == ("LoadOverlapped" if kernel == "k_step_dev" else "LoadReadOnly"), kernel


def test_overlapped_launches_are_those_known_here():
    for name in sorted(os.listdir(CSRC)):
        src = code(name)
        if "launch_pdl(" in src:
            assert name in REACHED, name
        assert "launch_pdl(k_step_batch" not in src, name
