"""The checked build on the kernel forms of production sizes.

Large calls take other forms of the kernels than the small ones of
test_gpu_checked.py: two resident CTAs per SM, two expert-body streams per CTA, 16
epilogue warps, and groups of eight sequence blocks.  Each shape here is the
smallest that takes its form; no check fails, and the results agree with the
default build's."""
import numpy as np
import pytest

import test_gpu_checked as tc
from test_gpu_checked import checked_path  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

CASES = {
    # more than 152 (expert, probe) pairs
    "resident_two_per_sm": tc._lstm_step((2, 32, 48, 16, 5, 80)),
    "resident_two_per_sm_sparse": tc._lstm_step((1, 16, 24, 5, 6, 200), kind="sparse"),
    # probe tiles in shared memory
    "resident_shared_tiles": tc._lstm_step((1, 32, 64, 16, 4, 3)),
    # more than 152 tasks of more than two chunks, three stages
    "persistent_wide_p1": tc._lstm_step((1, 16, 100, 40, 4, 100)),
    "persistent_wide_p2_sparse": tc._lstm_step((1, 16, 100, 30, 4, 101), kind="sparse"),
    # more than 152 tasks of eight blocks; the last group of one block of one sequence
    "eval_eight_blocks": tc._eval((40, 16, 66, 257, 4)),
    "eval_odd_blocks": tc._eval((40, 16, 66, 70, 3)),
    "mixture_eight_blocks": tc._mixture(N=30, E=16, H=66, R=900, k=2, T=5, t0=1),
    # more than 152 streams, an odd number per expert
    "body_two_streams": tc._body(N=1, n=81, B=20, T=5),
    "body_two_streams_odd": tc._body(D=1, N=3, n=67, B=4, T=5),
}


@pytest.mark.parametrize("name", list(CASES))
def test_no_check_fails_and_results_agree(checked_path, name):  # noqa: F811
    run = CASES[name]
    with tc.using(tc._default_path()) as a:
        want, _ = run(a)
        assert a.get_status() == 0
        want = tc._host(want)
    with tc.using(checked_path) as a:
        assert a.lib().soma_checked_build() == 1
        got, _ = run(a)
        status = a.get_status()
        line = a.lib().soma_debug_check_line(None)
        assert (status, line) == (0, 0), (a.STATUS_NAMES.get(status, status), line)
        got = tc._host(got)
    for k in want:
        np.testing.assert_allclose(got[k], want[k], rtol=1e-5, atol=1e-6, err_msg=k)
