"""The autotuner does not choose between block sizes that launch the same kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["CL_FP64", "CL_FP32_STORAGE", "CL_DF64"])
def test_sizes_of_one_launch_have_one_time(form):
    from paper_1311_1056_gb300 import cl

    cp = cl.make_cool(0.01, mode=cl.CL_D1, n_max=2)
    with cl.Lattice((6, 4, 4, 6), beta=6.0, theta=1.0, prec=getattr(cl, form), start=cl.CL_START_HOT) as lat:
        blocks, table = lat.autotune(0.01, cp, reps=2, use_cache=False, want_table=True)
    for fam in (3, 4):  # the cooling kernels' one shape
        assert np.all(table[:, fam] == table[0, fam]) and blocks[fam] == 128
    if form != "CL_FP32_STORAGE":  # link algebra: at most 128 threads
        assert np.array_equal(table[3, :2], table[2, :2]) and max(blocks[:2]) <= 128
