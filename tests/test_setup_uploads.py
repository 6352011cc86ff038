"""An executor's tables (leaves, gathers, permutation, runs of small steps) are
uploaded from pageable memory, which returns before the copy has reached the
device; a call's stream may be a non-blocking one, which does not wait for the
stream of the copies.  So the set-up has to wait for them before it returns.
Checked on the source: the window is far too short to meet by running."""
import os


def test_setup_waits_for_its_copies():
    from paper_2110_14502_gb300 import build as B
    with open(os.path.join(B.CSRC, "executor.cu")) as f:
        text = f.read()
    at = text.index("static tn_status setup(Plan& P, Executor& E) {")
    body = text[at:text.index("\n}\n", at)]
    last = body.rindex("cudaMemcpy(")
    assert "CK(cudaStreamSynchronize(nullptr));" in body[last:], body[last:]
