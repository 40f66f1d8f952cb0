"""The tensor-core level-0 kernel when one of its bounded waits runs out, read from the source: it ends the copies of A it
has started and every MMA it has issued, each with a limit, before it gives tensor memory back and returns."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_07656_gb300", "csrc", "k_corr0_tc.cu")


def test_in_flight_work_ends_first():
    s = re.sub(r"//[^\n]*", "", open(SRC).read())
    kernel = s[s.index("k_corr0_tc(const __grid_constant__"):]
    out = kernel[kernel.index("if (*abort_flag) break;"):kernel.index("tcgen05.dealloc")]
    a, m = out.index("mbar_drain(bar_full"), out.index("tcgen05.commit")
    assert "if (*abort_flag) {" in out[:a] and "mbar_drain(bar_gone, 0);" in out[m:]
    assert out.rindex("__syncthreads();") > max(a, m)
    # every copy is counted where it is issued, and the drain's wait has a limit and no early way out
    assert re.search(r"cp\.async\.bulk\.shared::cluster\.global[^;]*;[^;]*;?\s*issued = it \+ 1;", kernel)
    drain = s[s.index("void mbar_drain("):]
    drain = drain[:drain.index("\n}")]
    assert "<= WAIT_CYCLES" in drain and "abort" not in drain
