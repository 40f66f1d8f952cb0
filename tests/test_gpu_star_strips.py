"""DM*'s entry points where the split of a map changes: widths of level 1 at, just below and
just past one and two strips of 62 columns, heights at and past a work item's 32 rows, one-
and two-pixel rests; matches bit for bit against the FP32 oracle, both child sums."""
import numpy as np
import pytest

import oracle
from paper_1506_07656_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compensated", [True, False])
@pytest.mark.parametrize("W2,H2", [(122, 34), (123, 64), (125, 65), (126, 30), (248, 67), (249, 36), (19, 130)])
def test_entries_bit_exact(W2, H2, compensated):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    a = synth.make_pair_smooth(36, 28, W2).img1.astype(np.float32)
    b = synth.make_pair_smooth(W2, H2, H2).img2.astype(np.float32)
    ctx = dm.Context(dm.DM_FP32, compensated=compensated)
    try:
        got = ctx.match_star(a, b).cpu().numpy()
    finally:
        ctx.close()
    want = oracle.dmstar_match(a, b, "f32", compensated=compensated).astype(np.float32)
    np.testing.assert_array_equal(got, want)
