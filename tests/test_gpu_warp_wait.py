"""A bounded wait gives one answer to the whole warp.

After a wait that runs out, a warp leaves its loop; lanes that left alone would
be waited for, without a bound, by the shuffles and tensor-memory loads of the
others.  Here the lanes of a warp disagree by construction: half of them wait
on a barrier that nothing completes."""
import pytest

from gpu_common import api

pytestmark = pytest.mark.gpu

SOMA_ERR_TIMEOUT = 5


@pytest.mark.parametrize("mixed,polls", [(False, 1), (False, 1000), (True, 1), (True, 63),
                                         (True, 1000)])
def test_every_lane_gets_the_same_answer(mixed, polls):
    a = api()
    assert a.get_status() == 0
    got = a.debug_warp_wait(mixed, polls)
    assert a.get_status() == (SOMA_ERR_TIMEOUT if mixed else 0)
    assert got.tolist() == [0 if mixed else 1] * 32
