"""The spreading launch that a plan chooses (host.cu: spread_shape), on the limits of a GB300, for every size a plan
takes: it fits the block, and the block's warps do not dwindle where a grid nearly fills it."""
import itertools
import math

import pytest

from _host_program import host_program

# shared memory per block (opt-in), per SM, reserved per block; SMs, threads per SM
LIMITS = (232448, 233472, 1024, 152, 2048)
PROGRAM = """
int main()
{
    int d, N, M, w, f32, ang, thr, per;
    double sigma;
    while (scanf("%d %d %d %d %lf %d %d %d %d", &d, &N, &M, &w, &sigma, &f32, &ang, &thr, &per) == 9) {
        pgbh::SpreadShape s{};
        const int nf = pgbh::grid_size(N, sigma) / 2 + 1;
        const int rc = pgbh::spread_shape({d, N, M, nf, w, f32 != 0, ang != 0, thr, per, LIMITS}, s);
        printf("%d %d %d %d %d %zu %d %d %lld %d\\n", rc, s.nslab, s.rows_per_slab, s.threads, s.blocks, s.smem, s.queued,
               s.nsplit, s.nitem, nf);
    }
}
"""
PROGRAM = PROGRAM.replace("LIMITS", ", ".join(map(str, LIMITS)))


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("shape"), PROGRAM)
    keys = ("rc", "nslab", "rows", "threads", "blocks", "smem", "queued", "nsplit", "nitem", "nf")

    def shapes_of(plans):
        text = "".join("%d %d %d %d %.17g %d %d %d %d\n" % p for p in plans)
        return [dict(zip(keys, map(int, line.split()))) for line in run(stdin=text)]
    return shapes_of


def _plans(f32, threads=0):
    widths = range(2, 11) if f32 else range(2, 17)
    for w, sigma, ang in itertools.product(widths, (1.5, 2.0, 4.0), (0, 1)):
        for N in range(2, 160):
            yield (2, N, 8, w, sigma, int(f32), ang, threads, 0)
        for N in range(2, 40):
            yield (3, N, 8, w, sigma, int(f32), ang, threads, 0)


@pytest.mark.parametrize("f32", [True, False])
def test_every_plan_fits_and_is_covered(shapes, f32):
    plans = list(_plans(f32))
    for p, s in zip(plans, shapes(plans)):
        if s["rc"]:
            continue
        assert s["smem"] <= LIMITS[0] - 1024 and 32 <= s["threads"] <= (640 if f32 else 512), (p, s)
        assert s["threads"] % 32 == 0 and s["blocks"] % s["nslab"] == 0, (p, s)
        assert (s["nslab"] - 1) * s["rows"] < s["nf"] <= s["nslab"] * s["rows"], (p, s)


def test_fp32_blocks_keep_their_warps(shapes):
    """At least 320 threads (3D 384) with their queues, one slab or several, unless the plan is too small for them or a
    single plane of the grid leaves no room."""
    plans = list(_plans(True))
    for p, s in zip(plans, shapes(plans)):
        d, N, M, w = p[:4]
        classes = (N * (N + 1) // 2) ** d * s["nsplit"]
        least = min(320 if d == 2 else 384, max(64, math.ceil(classes / 152)))
        if s["rc"] or s["rows"] == 1:
            continue
        assert s["queued"] or s["nslab"] > 1, (p, s)
        assert s["threads"] >= least, (p, s)


def test_fp64_2d_small_plans_share_their_quads(shapes):
    """A thread adds the 16 points of an orbit's quad one after the other only where there are quads for a quarter
    of the GPU's threads; below that they are cut into 4 shares or 16 (one point each; 8 points at M = 4: 16 or none)."""
    plans = [(2, N, M, w, 2.0, 0, ang, 0, 0) for N in range(2, 65) for M in (2, 4, 6, 12, 32) for w in (6, 10, 14) for ang in (0, 1)]
    for p, s in zip(plans, shapes(plans)):
        N, M = p[1:3]
        norb = sum(1 for i in range(N) for j in range(i, N) if i + j <= N - 1)
        if not s["queued"]:
            assert M == 2 and s["nsplit"] == 1 and (N * (N + 1) // 2) ** 2 <= 152 * 512 * 2 // 3, (p, s)
            continue
        quads = norb ** 2 * (M // 4 + 1)
        assert s["nitem"] == quads * s["nsplit"] and s["nsplit"] in (1, 4, 16), (p, s)
        assert s["nsplit"] > 1 or (4 if M > 4 else 24) * quads > 152 * 512, (p, s)


def _accepted_before(d, w, nf, f32, threads):
    """Whether a plan with points spread one by one through queues of 2 d + 1 floats (FP64: d + 1 doubles) per thread, with
    a margin column more on both sides of the last axis (and padded FP64 3D tiles), found room for a row of the grid."""
    room = LIMITS[0] - 1024 - 16 - (0 if f32 else 8 * 136)
    plane = nf ** (d - 2) * (nf + 2 * (w // 2 + 1)) * (4 if f32 else 12)
    queue = threads * (4 * (2 * d + 1) if f32 else 8 * (d + 1))
    return nf * plane <= room or queue + plane <= room


@pytest.mark.parametrize("threads", [32, 64, 96, 128, 256, 1024])
def test_no_block_size_is_refused_that_was_not_before(shapes, threads):
    """3D FP32 grids whose planes all but fill the block: the queues per thread grew, the block shrinks instead."""
    plans = [(3, N, 4, w, sigma, 1, ang, threads, 0) for w in range(2, 11) for sigma in (1.5, 2.0, 4.0) for ang in (0, 1)
             for N in range(2, 129)]
    for p, s in zip(plans, shapes(plans)):
        if _accepted_before(3, p[3], s["nf"], True, threads):
            assert s["rc"] == 0 and s["threads"] <= threads and s["smem"] <= LIMITS[0] - 512, (p, s)


BATCH = """
int main()
{
    int d, f32, ask, automatic;
    long long tile, limit;
    while (scanf("%d %d %d %d %lld %lld", &d, &f32, &ask, &automatic, &tile, &limit) == 6)
        printf("%d\\n", pgbh::batch_block_threads(d, f32 != 0, ask, automatic, tile, limit));
}
"""


def test_batched_blocks_that_are_asked_for(tmp_path):
    """Refused exactly when 2 d + 1 floats per thread do not fit beside the tile (FP64: when the tile does not); otherwise
    the largest block up to the one asked for whose queues fit."""
    run, limit = host_program(tmp_path, BATCH), 230000
    cases = [(d, f32, ask, 128, limit - left, limit) for d in (2, 3) for f32 in (0, 1) for ask in (32, 96, 256, 512, 1024)
             for left in (0, 1000, 2000, 3000, 6000, 12000, 13000, 24000, 28000, 40000)]
    out = run(stdin="".join("%d %d %d %d %d %d\n" % c for c in cases))
    for (d, f32, ask, _, tile, _), got in zip(cases, map(int, out)):
        left = limit - tile
        if not f32:
            assert got == min(ask, 512)
            continue
        per = {2: 44, 3: 68}[d]
        fits = min(ask, 640, left // (32 * per) * 32)
        assert got == (fits if ask * 4 * (2 * d + 1) <= left else 0), (d, ask, left, got)
