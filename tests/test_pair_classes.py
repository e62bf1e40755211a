"""The spreading kernels' classes of node pairs (spread_impl.cuh: PairData, PairCursor): host checks
of the numbering and of the class strengths against the ordered double sum, and on the GPU the
independence of the result from the launch shape (every class is spread exactly once)."""
import itertools
import random

import numpy as np
import pytest

K = 1597  # the row shear of the class numbering (kPairShear)


def _axis_pair(p, N):
    t = int((np.float32(p) + np.float32(0.5)) * (np.float32(1.0) / np.float32(N)))
    u = p - t * N
    return u, (u + t) % N, t


def test_axis_pairs_cover_every_unordered_pair_once():
    for N in list(range(2, 40)) + [63, 64, 120, 121, 200, 511, 512]:
        seen = {tuple(sorted(_axis_pair(p, N)[:2])) for p in range(N * (N + 1) // 2)}
        assert len(seen) == N * (N + 1) // 2, N


@pytest.mark.parametrize("d,N", [(2, 2), (2, 3), (2, 4), (2, 7), (3, 2), (3, 3), (3, 4)])
def test_class_strengths_sum_to_the_ordered_double_sum(d, N):
    """For every centre and radius: 2 prod(1/2 on equal axes) sum over the 2^(d-1) exchanges equals
    the sum of a_i a_j over the ordered pairs that have them, and cos theta changes sign on the
    exchanged axes."""
    rng = np.random.default_rng(d * 10 + N)
    v = np.sort(rng.normal(size=N))  # no accidental coincidences
    a = rng.normal(size=(N,) * d)
    want = {}
    nodes = list(itertools.product(range(N), repeat=d))
    for i in nodes:
        for j in nodes:
            key = tuple(tuple(sorted((x, y))) for x, y in zip(i, j))
            want[key] = want.get(key, 0.0) + a[i] * a[j]
    naxp = N * (N + 1) // 2
    got = {}
    for pr in range(naxp ** d):
        t, u = divmod(pr, naxp)
        ap = [t] if d == 2 else list(divmod(t, naxp))
        ap.append((u + t * K) % naxp)
        ni, nj, rows = zip(*(_axis_pair(p, N) for p in ap))
        x = 0.0
        for o in range(1 << (d - 1)):
            I = tuple(nj[l] if (o >> l) & 1 else ni[l] for l in range(d))
            J = tuple(ni[l] if (o >> l) & 1 else nj[l] for l in range(d))
            x += a[I] * a[J]
            assert np.allclose([abs(v[q] - v[w]) for q, w in zip(I, J)], [abs(v[q] - v[w]) for q, w in zip(ni, nj)])
        got[tuple(tuple(sorted(z)) for z in zip(ni, nj))] = 2.0 * 0.5 ** sum(r == 0 for r in rows) * x
    assert got.keys() == want.keys()
    assert all(abs(got[k] - want[k]) < 1e-12 for k in want)


def test_class_cursor_matches_the_numbering():
    rng = random.Random(11)
    for _ in range(1500):
        N = rng.choice([2, 3, 16, 64, 120, 512, rng.randint(2, 512)])
        n = N * (N + 1) // 2
        total = n ** rng.choice([2, 3])
        stride = rng.choice([1, 64, 1024, 152 * 1024, rng.randint(1, 10 ** 6)])
        pr = rng.randint(0, min(total - 1, 10 ** 9))
        t, u = divmod(pr, n)
        i = (u + t * K) % n
        dt, du = divmod(stride, n)
        di, dk = (du + dt * K) % n, K % n
        for _ in range(40):
            if pr >= total:
                break
            assert (t, u, i) == (*divmod(pr, n), (pr % n + pr // n * K) % n)
            pr, t, u, i = pr + stride, t + dt, u + du, i + di
            if i >= n:
                i -= n
            if u >= n:
                u, t, i = u - n, t + 1, i + dk
                if i >= n:
                    i -= n


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [1, 2])  # PG_PREC_FP64, PG_PREC_FP32
@pytest.mark.parametrize("d,N,M,ang", [(2, 2, 2, None), (2, 9, 6, None), (2, 16, 8, [1.0, 0.5, 0.3]), (3, 2, 4, None),
                                       (3, 5, 6, None), (3, 5, 8, [1.0, 0.0, 0.4])])
def test_result_does_not_depend_on_the_launch_shape(d, N, M, ang, prec):
    """Exact integer accumulation: the same bits for every block size and block count (FP64 rounds
    each block's cell sums to the grid unit, 2^-60 of the strength bound)."""
    import torch
    from paper_2105_08806_gb300 import Plan
    rng = np.random.default_rng(N)
    f = torch.as_tensor(rng.normal(size=(N + 1) ** d) * 0.1, device="cuda")
    out = []
    for threads, per_sm in ((0, 0), (32, 1), (96, 2), (256, 1)) + (((1024, 1),) if prec == 2 else ()):
        Q = torch.empty_like(f)
        with Plan(d, N, M, 2.0, 0.5, 1e-6, precision=prec, angular=ang, spread_threads=threads,
                  spread_blocks_per_sm=per_sm) as plan:
            plan.collide(f, Q)
            torch.cuda.synchronize()
        out.append(Q.cpu().numpy())
    for q in out[1:]:
        if prec == 2:
            assert np.array_equal(q, out[0])
        else:
            assert np.abs(q - out[0]).max() <= 1e-12 * np.abs(out[0]).max()
