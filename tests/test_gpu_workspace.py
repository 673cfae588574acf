"""A workspace asked for at some counts serves every call with counts that are no larger: C callers hold one for the
largest counts that they will have."""
import itertools

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# about every line where a plan changes form
COUNTS = [1, 129, 1_280, 8_000, 10_700, 11_999, 12_000, 15_999, 16_000, 16_383, 16_384, 16_385, 20_011, 46_000, 60_000,
          131_072, 200_000, 262_144, 1_000_000, 2_900_000, 2_965_000, 3_100_000, 5_000_000]
SEGMENTS = [0, 640, 1_024, 1_028, 5_120, 40_000]


@pytest.fixture(scope="module")
def size():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_11430_gb300 import _lib, api, build

    build.build()
    memo = {}

    def f(op, *a):
        if (op,) + a not in memo:
            memo[(op,) + a] = api.workspace_size(getattr(_lib, op), *a)
        return memo[(op,) + a]

    return f


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("op", ["VPM_OP_INDUCE", "VPM_OP_BACKWARD"])
def test_sources_and_targets(size, op, flags):
    for a, b in itertools.product(range(len(COUNTS)), repeat=2):
        here = size(op, COUNTS[a], COUNTS[b], 0, flags)
        if a:
            assert size(op, COUNTS[a - 1], COUNTS[b], 0, flags) <= here, (COUNTS[a], COUNTS[b])
        if b:
            assert size(op, COUNTS[a], COUNTS[b - 1], 0, flags) <= here, (COUNTS[a], COUNTS[b])


@pytest.mark.parametrize("flags", [0, 1, 3])
@pytest.mark.parametrize("op", ["VPM_OP_RHS", "VPM_OP_STEP", "VPM_OP_STAGE", "VPM_OP_RHS_TREE", "VPM_OP_STEP_TREE"])
def test_particles_and_segments(size, op, flags):
    for a, b in itertools.product(range(len(COUNTS)), range(len(SEGMENTS))):
        here = size(op, COUNTS[a], 0, SEGMENTS[b], flags)
        if a:
            assert size(op, COUNTS[a - 1], 0, SEGMENTS[b], flags) <= here, (COUNTS[a], SEGMENTS[b])
        if b:
            assert size(op, COUNTS[a], 0, SEGMENTS[b - 1], flags) <= here, (COUNTS[a], SEGMENTS[b])


@pytest.mark.parametrize("flags", [0, 1])
def test_segments_and_targets(size, flags):
    for a, b in itertools.product(range(len(COUNTS)), range(1, len(SEGMENTS))):
        here = size("VPM_OP_SEGMENTS", 0, COUNTS[a], SEGMENTS[b], flags)
        if a:
            assert size("VPM_OP_SEGMENTS", 0, COUNTS[a - 1], SEGMENTS[b], flags) <= here, (COUNTS[a], SEGMENTS[b])
        assert size("VPM_OP_SEGMENTS", 0, COUNTS[a], SEGMENTS[b - 1], flags) <= here, (COUNTS[a], SEGMENTS[b])
