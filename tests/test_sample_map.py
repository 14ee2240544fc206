"""Launch shapes of rows of few samples (host arithmetic, no GPU): on large
launches a lane takes up to four single samples, so that few lanes of a node
stay idle; 16-byte rows keep at least two lanes."""
import pytest

LARGE = 1023 * 1023 // 2


@pytest.fixture(scope="module")
def sample_map():
    from paper_2302_13680_gb300 import build

    build.build()
    from paper_2302_13680_gb300.cmg import sample_map

    return sample_map


@pytest.mark.parametrize("N,elem,expected", [
    (1, 4, (1, 1, 1)), (2, 4, (1, 1, 2)), (3, 4, (1, 1, 4)), (5, 4, (2, 1, 4)), (6, 4, (2, 1, 4)), (7, 4, (2, 1, 4)),
    (9, 4, (4, 1, 4)), (15, 4, (4, 1, 4)), (4, 4, (1, 4, 1)), (8, 4, (2, 4, 1)), (12, 4, (2, 4, 2)), (16, 4, (2, 4, 2)),
    (1, 8, (1, 1, 1)), (2, 8, (1, 2, 1)), (3, 8, (1, 1, 4)), (5, 8, (2, 1, 4)), (7, 8, (4, 1, 2)), (9, 8, (4, 1, 4)),
    (4, 8, (2, 2, 1)), (6, 8, (2, 2, 2)), (8, 8, (2, 2, 2))])
def test_few_samples_on_large_grids(sample_map, N, elem, expected):
    assert sample_map(N, elem, LARGE) == expected


@pytest.mark.parametrize("elem", [4, 8])
@pytest.mark.parametrize("items", [0, 9, 500, 8000, 32512, LARGE])
def test_every_count_is_covered(sample_map, elem, items):
    for N in range(1, 257):
        lanes, width, chunks = sample_map(N, elem, items)
        assert lanes * width * chunks >= N and N % width == 0
        assert lanes & (lanes - 1) == 0 and lanes <= 32 and chunks & (chunks - 1) == 0 and chunks <= 8
