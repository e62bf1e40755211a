"""Launch shapes that the batched autotuner times (host.cuh: tune_shapes): the current one first and the one the plan
started with, whatever they are, so that a tuned plan is no slower than before; the others within the limits."""
import pytest

from _host_program import host_program

PROGRAM = """
int main(int, char **a)
{
    const int limit = atoi(a[7]);  // threads per SM that the made-up occupancy allows; no block above `limit` fits
    for (const pgbh::LaunchShape &s : pgbh::tune_shapes({atoi(a[1]), atoi(a[2])}, {atoi(a[3]), atoi(a[4])}, 152, atoi(a[5]),
                                                        atoll(a[6]), [&](int t) { return limit / t; }))
        printf("%d %d\\n", s.threads, s.blocks);
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("tune"), PROGRAM)
    return lambda *args: [tuple(map(int, line.split())) for line in run(args)]


@pytest.mark.parametrize("now,start,most,limit", [((640, 152), (640, 152), 152, 640), ((96, 152), (96, 152), 152, 96),
                                                  ((512, 152), (640, 152), 152, 640), ((192, 760), (192, 760), 10 ** 9, 1024)])
def test_current_and_first_shapes_are_timed(shapes, now, start, most, limit):
    out = shapes(*now, *start, 640, most, limit)
    assert out[0] == now and start in out and len(set(out)) == len(out)
    for threads, blocks in out:
        assert (threads, blocks) in (now, start) or (threads in (128, 256, 512) and blocks % 152 == 0 and
                                                     blocks <= most and threads * blocks // 152 <= limit)
    assert {t for t, _ in out} >= {t for t in (128, 256, 512) if t <= limit}
