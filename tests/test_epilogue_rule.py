"""The persistent kernel's choice of 8 or 16 epilogue warps (host arithmetic).

Sixteen warps pay only where a task has more 8-sequence chunks than two groups of
warps can take.  With one or two chunks the wider form has warps without a share,
and those sweeps ran up to 10 % slower with it than with eight."""
import pytest

from paper_2609_37899_gb300 import api, build

DENSE, SPARSE = 0, 1


@pytest.fixture(scope="module")
def warps():
    build.build()
    return lambda N, E, H, n, kind, B: api.lib().soma_debug_epilogue_warps(
        api.dims(E, H), N, n, kind, B, 152)


@pytest.mark.parametrize("kind", [DENSE, SPARSE])
@pytest.mark.parametrize("N,E,H,n,B", [
    (8, 64, 66, 64, 1),      # two probes of one chunk each
    (8, 64, 200, 64, 4),
    (4, 64, 300, 64, 8),
    (8, 64, 400, 32, 8),
    (1, 16, 100, 128, 7),
    (64, 64, 66, 1, 8),      # one probe of one chunk
    (64, 64, 300, 1, 16),    # of two
])
def test_no_warps_without_a_share(warps, N, E, H, n, B, kind):
    assert warps(N, E, H, n, kind, B) == 8


@pytest.mark.parametrize("S,chunks4,chunks8", [  # stages, with 4 and with 8 chunks
    (3, (16, 16), (16, 16)), (4, (16, 16), (16, 16)), (5, (16, 8), (16, 16)),
    (6, (8, 8), (16, 16)), (8, (8, 8), (16, 8)), (9, (8, 8), (8, 8)), (16, (8, 8), (8, 8))])
def test_stages(warps, S, chunks4, chunks8):
    H = 64 * (S - 1)
    for B, want in ((16, chunks4), (32, chunks8), (64, chunks8)):
        assert (warps(8, 64, H, 64, DENSE, B), warps(8, 64, H, 64, SPARSE, B)) == want


def test_few_tasks_and_invalid_sizes(warps):
    assert warps(1, 16, 100, 50, DENSE, 32) == 8    # 150 tasks
    assert warps(1, 16, 100, 51, DENSE, 32) == 16   # 156
    assert warps(1, 16, 100, 64, DENSE, 65) == 0
    assert warps(0, 16, 100, 64, DENSE, 8) == 0
