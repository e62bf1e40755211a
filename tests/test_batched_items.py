"""Work items of batched plans (host.cuh: default_item_points): a few small cells make as many items of classes of node
pairs as they would of single pairs at 2^17 points each, so that the SMs share them as evenly."""
import pytest

from _host_program import host_program

PROGRAM = """
int main(int, char **a) { printf("%lld\\n", pgbh::default_item_points(atoi(a[1]), atoll(a[2]), atoi(a[3]))); }
"""


@pytest.mark.parametrize("d,cells", [(2, [(16, 8), (24, 8), (24, 16), (16, 16)]), (3, [(6, 8), (8, 16), (10, 8), (6, 16)])])
def test_items_of_classes_are_as_many_as_of_pairs(tmp_path, d, cells):
    run = host_program(tmp_path, PROGRAM)
    count = lambda n, size, M: -(-n // max(64, size // M))  # noqa: E731
    classes = lambda item: sum(count((N * (N + 1) // 2) ** d, item, M) for N, M in cells)  # noqa: E731
    pairs = sum(count(N ** d * (N ** d + 1) // 2, 1 << 17, M) for N, M in cells)
    item = int(run([d, classes(1 << 17), 152])[0])
    assert classes(item) >= pairs
    assert int(run([d, 2 * 152, 152])[0]) == 1 << 17  # many items: whole ones
