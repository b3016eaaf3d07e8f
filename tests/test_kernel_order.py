"""Order of the synchronising instructions inside the kernels, read from their
source: what a run cannot show, because it comes out right by timing."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_08779_gb300", "csrc")


def kernel_text(file, name):
    """The body of the function `name` in csrc/`file`, without comments."""
    with open(os.path.join(CSRC, file)) as f:
        src = f.read()
    src = re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", src), flags=re.S)
    start = src.index("{", src.index(" " + name + "("))
    depth = 0
    for i in range(start, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[start:i + 1]
    raise AssertionError("unbalanced braces")


def test_cluster_gemv_waits_for_its_peers_before_remote_stores():
    # another CTA's shared memory exists only once that CTA has started: every
    # thread arrives at the cluster barrier on entry and waits for it before
    # the first store into a peer
    body = kernel_text("gemv_cluster.cu", "gemv_cluster_kernel")
    arrive = body.index("barrier.cluster.arrive.relaxed.aligned")
    wait = body.index("barrier.cluster.wait.acquire.aligned")
    assert arrive < wait < body.index("st.shared::cluster")
    assert wait < body.index("cluster.sync()")


@pytest.mark.parametrize("file,name", [
    ("gemv_cluster.cu", "gemv_cluster_kernel"),
    ("gemv_batch.cu", "gemv_batch_kernel"),
    ("quantize.cu", "quantize_kernel"),
    ("quantize.cu", "rotate_rows_ring"),
    ("quantize.cu", "hadamard_rows_kernel"),
])
def test_the_next_kernel_starts_only_behind_the_wait(file, name):
    # a sss_gemv_multi with SSS_GEMV_WEIGHTS_READY reads its weights as soon as it
    # starts: were it let in before this kernel's wait, they might still be being
    # written by the launch before this one
    body = kernel_text(file, name)
    assert body.index("griddepcontrol.wait") < body.index("griddepcontrol.launch_dependents")


def test_the_streaming_gemv_lets_the_next_kernel_in_early_only_with_early_weights():
    body = re.sub(r"\s+", " ", kernel_text("gemv_stream.cu", "gemv_stream_kernel"))
    release = 'asm volatile("griddepcontrol.launch_dependents;" ::: "memory");'
    assert body.count(release) == 2
    assert "if (a.early_weights) " + release in body
    assert 'if (!a.early_weights) { asm volatile("griddepcontrol.wait;" ::: "memory"); ' + release in body


@pytest.mark.parametrize("name", ["hadamard_rows_kernel", "hadamard_cols_kernel"])
def test_the_rotation_without_a_status_has_no_wait_that_can_expire(name):
    # sss_hadamard takes no status word: an expired wait would go unreported
    body = kernel_text("quantize.cu", name)
    for called in ("q_wait", "rotate_rows_ring", "mbarrier"):
        assert called not in body
