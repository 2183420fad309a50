"""The restricted chain against its float64 oracle with windows that reach a part of a block of 64 loci: within a
half, across the halves' and the blocks' borders, for every slots-per-lane variant."""
import pytest

from tests.test_gpu_sparse_blocks import ls, test_blocks_and_slots as check  # noqa: F401  (ls: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,WS,K,lookahead,mu,pool", [
    (20, 140, 1, 5, 0, 1e-3, True), (20, 140, 7, 5, 1, "locus", True), (24, 140, 16, 9, 0, 0.7, True),
    (24, 140, 31, 9, 2, 1e-3, True), (24, 140, 32, 9, 0, "locus", True), (24, 140, 33, 9, 0, 1e-3, False),
    (24, 200, 48, 9, 1, 1e-3, True), (24, 200, 65, 9, 0, "locus", True), (24, 200, 96, 9, 2, 1e-3, True),
    (110, 100, 20, 100, 0, 1e-3, True), (150, 70, 9, 66, 2, "locus", True), (310, 40, 17, 300, 0, 1e-2, True),
    (400, 70, 40, 390, 1, 1e-2, True), (460, 70, 35, 450, 2, 1e-2, True)])
def test_windows_within_blocks(ls, N, L, WS, K, lookahead, mu, pool):  # noqa: F811
    check(ls, N, L, WS, K, lookahead, mu, pool)
