"""Workspace queries (host only): a workspace for n points is enough for every
smaller n.  Callers rely on it, and so does the library: lap_run_full sizes
its scratch for all n points once and takes the column means of every level's
subset in it."""
import pytest

from paper_0910_1650_gb300 import build as b
from paper_0910_1650_gb300 import capi


@pytest.fixture(scope="module")
def lib():
    b.build()
    return capi.lib()


def _never_shrinks(query, sizes):
    largest = 0
    for n in sizes:
        need = query(n)
        assert need >= largest, n
        largest = need


@pytest.mark.parametrize("d", [1, 64, 129, 300, 4096])
def test_point_set_queries_never_shrink(lib, d):
    """The column sums' row blocks are fewer at many larger sizes (d = 64: 152 at
    4864 points, 148 at 4865); the scratch must not follow them down.  Sizes to
    10000 one by one, and around the 2048-block limit."""
    near = [w * 2048 + e for w in (255, 256, 257, 263, 264, 300) for e in (-1, 0, 1)]
    for sizes in (range(2, 10001), near):
        _never_shrinks(lambda n: lib.lap_assign_workspace_size(n, d, 2), sizes)
        _never_shrinks(lambda n: lib.lap_refine_workspace_size(n, d, 2), sizes)
        _never_shrinks(lambda n: lib.lap_run_full_workspace_size(n, d, 2, 2, 2), sizes)
        _never_shrinks(lambda n: lib.ap_similarity_workspace_size(n, d), sizes)


def test_training_query_never_shrinks(lib):
    """A training loop's last batch is the smallest.  The partial sums of W2's
    gradient are fewer at many larger batches (38 at 1216 rows, 26 at 1217)."""
    _never_shrinks(lib.apl_workspace_size, range(1, 25001))


@pytest.mark.parametrize("d,c,row", [(300, 10, 644), (300, 1000, 644), (64, 768, 132), (128, 512, 260),
                                     (128, 513, 260), (64, 769, 148), (128, 1024, 276), (256, 1024, 516)])
def test_assignment_query_counts_the_groups_there_are(lib, d, c, row):
    """Per point: the bf16 features (d rounded up to 64), the choice, and 8 bytes
    for each group of CTAs the centres are dealt to where there are two (769 to
    1024 centres of up to 128 features)."""
    n = 1000000
    grow = lib.lap_assign_workspace_size(2 * n, d, c) - lib.lap_assign_workspace_size(n, d, c)
    assert abs(grow / n - row) < 0.1
