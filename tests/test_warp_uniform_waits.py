"""A bounded wait can end differently for the lanes of a warp (one sees the phase,
the next the other warps' failure), and the tensor-memory instructions take all
32 lanes: in the tensor-core kernels no lane may leave a loop, or reach tcgen05,
on its own wait's result alone.  Checked on the source: a wait's result is stored
or voted on (__all_sync, __syncthreads_and), never branched on directly, and the
result that guards a tensor-memory load has been voted on."""
import os
import re

from paper_1812_00118_gb300 import build as B

SRC = open(os.path.join(B.CSRC, "lbm_surrogate.cu")).read()


def kernels():
    """(name, body) of the kernels that use tensor memory."""
    for m in re.finditer(r"__global__ void[^\n]*\n(\w+)\(|__global__ void (\w+)\(", SRC):
        i = SRC.index("{\n", m.end())
        depth, j = 0, i
        while True:
            depth += {"{": 1, "}": -1}.get(SRC[j], 0)
            j += 1
            if depth == 0:
                break
        body = re.sub(r"//[^\n]*", "", SRC[i:j])
        if "tc_ld16(" in body:
            yield m.group(1) or m.group(2), body


def test_waits_are_voted_on():
    found = dict(kernels())
    assert set(found) == {"conv_tc_kernel", "conv_row_kernel", "conv_flat_kernel", "conv_wgrad_row_kernel"}
    for name, body in found.items():
        assert not re.search(r"if \(!?\s*mbar_(wait_phase|wait_bounded|try)\(", body), name
        for m in re.finditer(r"tc_ld16\(", body):
            # the last decision before the load: a vote, or a shared flag read after a barrier
            before = body[:m.start()]
            votes = [before.rfind(s) for s in ("__all_sync(", "__syncthreads_and(", "if (!failed &&")]
            assert max(votes) > max(before.rfind("mbar_wait_phase("), before.rfind("wait_stage(")) - 60, name
