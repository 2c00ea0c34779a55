"""The expert body's choice of one or two streams per CTA (host arithmetic).

Only streams of one expert share a CTA: what counts is the rounds of CTAs over the
SMs, not the number of streams."""
import pytest

from paper_2609_37899_gb300 import api, build


@pytest.fixture(scope="module")
def streams():
    build.build()
    return lambda N, n, B: api.lib().soma_debug_body_streams(N, n, B, 152)


@pytest.mark.parametrize("N,n,B,want", [
    (152, 1, 16, 1),    # every stream has an SM
    (5, 12, 21, 1),
    (200, 1, 16, 1),    # one stream per expert: nothing to share
    (256, 1, 1, 1),
    (100, 3, 16, 1),    # 200 CTAs of two take two rounds, as 300 of one
    (52, 5, 16, 1),
    (153, 1, 16, 1),
    (1, 153, 16, 2),    # 77 CTAs in one round against two
    (77, 2, 16, 2),
    (160, 1, 48, 2),    # three rounds against four
    (256, 3, 16, 2),
    (256, 64, 16, 2),
    (256, 64, 64, 2),
    (0, 1, 1, 0),
])
def test_streams_per_cta(streams, N, n, B, want):
    assert streams(N, n, B) == want
