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
