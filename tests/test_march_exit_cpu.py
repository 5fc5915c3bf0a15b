"""The march's block and empty-box exits (march_exit), replayed on the CPU in binary32.

On every axis only the face ahead of the ray bounds the estimate, and a face on or beyond
the grid's border is not clipped to infinity (its crossing lies at or behind the ray's own
exit t1 up to rounding). Whenever the estimate is taken without the exact search, it must be
the first lattice sample outside the box, the box being the one the search uses, clipped at
the border. Rays that leave through the border, start on it or run along an axis (components
+0 and -0) are among the cases."""
import numpy as np
import pytest

from tests.test_box_exit_cpu import F, INF, _case, _exit_margin, _in_box, _lattice_t, _ulp_perturb


def _inverse(x, rng):
    return INF if x == 0 else _ulp_perturb(F(F(1.0) / x), rng)


@pytest.mark.parametrize("N,B,n_cases,mode", [(64, 8, 700, "random"), (1024, 32, 700, "adversarial"),
                                              (48, 2, 500, "near_start"), (1024, 32, 700, "border")])
def test_estimate_with_unclipped_faces_matches_the_lattice(N, B, n_cases, mode):
    rng = np.random.default_rng(N + n_cases)
    taken = 0
    while n_cases:
        c = _case(rng, N, B, "random" if mode == "border" else mode)
        if c is None:
            continue
        o, d, t0, t1, k, _, _ = c
        if mode == "border":                 # the last samples of a ray; sometimes along a face or an axis
            if rng.uniform() < 0.4:
                i = int(rng.integers(0, 3))
                d, o = d.copy(), o.copy()
                d[i] = F(0.0) if rng.uniform() < 0.5 else F(-0.0)
                o[i] = F(rng.choice([0.0, rng.uniform(0, N), N]))
                with np.errstate(divide="ignore"):
                    ta = [(F(-o[a]) / d[a], F(F(N) - o[a]) / d[a]) for a in range(3) if d[a] != 0]
                t0, t1 = F(max(0.0, *(min(p) for p in ta))), F(min(max(p) for p in ta))
                if not t0 < t1:
                    continue
            k = max(0, int(t1 - t0) - int(rng.integers(0, 2 * B)))
        t = _lattice_t(t0, k)
        if not t < t1:
            continue
        j = [min(max(int(np.floor(F(o[i] + F(t * d[i])))), 0), N - 1) for i in range(3)]
        D = int(rng.choice([1, 1, 2, 5, 32]))
        lo, hi, te = [0.0] * 3, [0.0] * 3, t1
        for i in range(3):
            b = j[i] // B
            bl, bh = (b - D + 1, b) if d[i] < 0 else (b, b + D - 1)
            lo[i] = -INF if bl <= 0 else F(bl * B)
            hi[i] = INF if (bh + 1) * B >= N else F((bh + 1) * B)
            face = F(bl * B if d[i] < 0 else (bh + 1) * B)
            with np.errstate(invalid="ignore"):
                x = F(F(face - o[i]) * _inverse(d[i], rng))
            te = te if np.isnan(x) else min(te, x)
        assert _in_box(o, d, t0, t1, k, lo, hi)
        K = F(F(te - t0) - F(0.5))
        n = F(np.ceil(K))
        half = F(F(0.5) - _exit_margin(d, t1, N))
        n_cases -= 1
        if n > k + 0.5 and abs(F(F(n - K) - F(0.5))) < half:
            taken += 1
            assert _in_box(o, d, t0, t1, int(n) - 1, lo, hi) and not _in_box(o, d, t0, t1, int(n), lo, hi), (k, n)
    assert taken > 50
