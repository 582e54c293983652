"""The rank vote's certified bounds from the sums it forms: Q = sum q_k^2 and P = sum p_0^2 over the components, in FP32
(q_k = p_k - p_0; two components a lane side by side for K <= 16), instead of sum_k |q_k| per component.

A component's spectrum errs by at most sqrt(2) (K + 3) u times sum |q_k| (m != 0) or sum |q_k| + K |p_0| (m = 0), so the
squared errors of the C 64 components sum to at most 2 ((K + 3) u)^2 times sum_d (sum_k |q_k|)^2 <= (K - 1) Q and
sum_d (sum_k |q_k| + K |p_0|)^2 <= 2 (K - 1) Q + 2 K^2 P (Cauchy-Schwarz, q_0 = 0).  Checked here: the kernel's text forms
these sums; their FP32 values with the kernel's 1 % dominate the exact sums of absolute values, also where
Cauchy-Schwarz is an equality (all |q_k| equal) and where only p_0 counts (q = 0); and the eigenvalues' FP32 errors lie
inside the bound made of them."""

import os
import re

import numpy as np
import pytest

from test_vote_bound import F, U, _fma32, _half_spectrum, _twiddles

SIGMA = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_23569_gb300", "csrc", "sigma.cu")


def test_the_kernel_forms_these_sums():
    with open(SIGMA) as f:
        src = re.sub(r"\s+", " ", f.read())
    assert "const float esq = (float)(K - 1) * vsum(qsq), e0sq = 2.f * fmaf((float)(K * K), vsum(p0sq), esq);" in src
    assert "const float dx0 = 1.4143f * (float)(K + 3) * U32 * sqrtf(e0s) * 1.01f;" in src
    assert "const float dx = 1.4143f * (float)(K + 3) * U32 * sqrtf(es) * 1.01f;" in src
    assert "const float bm = (2.f * sl * dd + dd * dd) * 1.01f + 16.f * U32 * lm + 1e-30f;" in src


def _groups(K, D, rng):
    yield rng.uniform(0.0, 255.0, (D, K))
    yield 200.0 + rng.normal(0.0, 1e-3, (D, K))
    yield np.where(np.arange(K) == 0, 0.0, 100.0) * np.ones((D, 1))                         # every |q_k| the same
    yield 30.0 + np.where(np.arange(K) == 0, 0.0, 50.0 * (-1.0) ** np.arange(K)) * np.ones((D, 1))
    yield np.repeat(rng.uniform(0.0, 765.0, (D, 1)), K, 1)                                    # q = 0
    yield np.where(np.arange(K)[None] == D % K, 255.0, 0.0) * (np.arange(D)[:, None] == 5)   # one pixel differs


def _butterfly(lanes):
    """The warp's sum: five levels, each lane adding its partner's value."""
    v = np.array(lanes, dtype=F)
    for o in (16, 8, 4, 2, 1):
        v = (v + v[np.arange(32) ^ o]).astype(F)
    return v[0]


def _lane_values(D, K):
    """Components of each lane in its order, with the half (0 or 1) that adds them up."""
    step = 64 if K <= 16 else 32
    return [[(d + h * 32, h) for d in range(lane, D, step) for h in range(step // 32)] for lane in range(32)]


def _sums(p, K, rows):
    """FP32 sums over the lanes of the products of `rows` (a list of a component's factors), as the kernel adds them."""
    lanes = []
    for comps in _lane_values(len(p), K):
        half = [F(0.0), F(0.0)]
        for d, h in comps:
            for x in rows(d):
                half[h] = _fma32(x, x, half[h])
        lanes.append(F(half[0] + half[1]) if K <= 16 else half[0])
    return lanes


@pytest.mark.parametrize("K", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("C", [1, 3])
def test_sums_dominate_the_absolute_values(C, K):
    D = 64 * C
    for p in _groups(K, D, np.random.default_rng(10 * K + C)):
        p = p.astype(F)
        q = (p - p[:, :1]).astype(F)
        esq = [F(F(K - 1) * s) for s in _sums(p, K, lambda d: q[d, 1:])]
        e0sq = [F(F(2.0) * _fma32(F(K * K), s, e)) for s, e in zip(_sums(p, K, lambda d: p[d, :1]), esq)]
        l1 = np.abs(q.astype(np.float64)).sum(1)
        l10 = l1 + K * np.abs(p[:, 0].astype(np.float64))
        assert np.sqrt(np.float64(_butterfly(esq))) * 1.01 >= np.sqrt((l1 ** 2).sum())
        assert np.sqrt(np.float64(_butterfly(e0sq))) * 1.01 >= np.sqrt((l10 ** 2).sum())


@pytest.mark.parametrize("K", [4, 16, 32])
def test_eigenvalues_lie_inside_their_bounds(K):
    D = 64
    tc, ts = _twiddles()
    for p in _groups(K, D, np.random.default_rng(K)):
        p = p.astype(F)
        q = (p - p[:, :1]).astype(F)
        spec = [_half_spectrum([F(v) for v in q[d]], K, tc, ts, F) for d in range(D)]
        esq = [F(F(K - 1) * s) for s in _sums(p, K, lambda d: q[d, 1:])]
        e0sq = [F(F(2.0) * _fma32(F(K * K), s, e)) for s, e in zip(_sums(p, K, lambda d: p[d, :1]), esq)]
        p64 = p.astype(np.float64)
        for m in range(K // 2 + 1):
            if m == 0:
                lam = _butterfly(_sums(p, K, lambda d: [_fma32(F(K), p[d, 0], spec[d][0][0])]))
            else:
                lam = _butterfly(_sums(p, K, lambda d: [spec[d][m][1], spec[d][m][0]]))
            dd = 1.4143 * (K + 3) * U * np.sqrt(np.float64(_butterfly(e0sq if m == 0 else esq))) * 1.01
            bound = (2.0 * np.sqrt(np.float64(lam) * 1.02) * dd + dd * dd) * 1.01 + 16.0 * U * np.float64(lam) + 1e-30
            x = p64 if m == 0 else p64 - p64[:, :1]  # lambda_m, m != 0, is the differences'
            exact = (np.abs(x @ np.exp(-2j * np.pi * m * np.arange(K) / K)) ** 2).sum()
            slack = 1e-13 * (np.abs(x).sum(1) ** 2).sum()  # the FP64 evaluation itself
            assert abs(np.float64(lam) - exact) <= bound + slack, (K, m)
