"""bfloat16 factors with a pack per node in the two-launch form, at the depths it is used for:
its rounding errors are those of the other schedules.  Reference: the anchored iteration (every
16th step the whole affine step, the others the bfloat16 matrices applied to w - w_a) in float64
with the factor's bfloat16 [Bbar; L] and Lambda / (2 p), on the CPU."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import harness as H
from tests.test_gpu_two_launch import _refused, two_launch

pytestmark = pytest.mark.gpu


def _null_basis(E):
    """The orthonormal null-space basis of E, by Householder reflections of E'."""
    M, n_e = E.T.copy(), E.shape[0]
    Q = np.eye(len(M))
    for k in range(n_e):
        v = np.zeros(len(M))
        v[k:] = M[k:, k]
        nrm = np.sqrt(v @ v)
        v[k] += nrm if M[k, k] > 0 else -nrm
        M -= (2 / (v @ v)) * np.outer(v, v @ M)
        Q -= (2 / (v @ v)) * np.outer(Q @ v, v)
    return Q[:, n_e:]


def _bf16(a):
    return torch.from_numpy(np.asarray(a, np.float64)).to(torch.bfloat16).double().numpy()


def _f32(a):
    return np.asarray(a, np.float32).astype(np.float64)


def _anchored(P, steps, iters, every, polish):
    """x of the anchored iteration with float32 constants and everything else in float64."""
    tree, f, cu = H.oracle_build(P)
    n, nx = tree.n, P["net"]["n_x"]
    L = _null_basis(P["net"]["E"])
    K = np.vstack([P["net"]["B"] @ L, L])
    Lam = -np.linalg.inv(L.T @ P["cost"]["W_u"] @ L)
    K16 = _bf16(K)
    L16 = np.stack([_bf16(Lam / (2 * p)) for p in tree.prob])
    L64 = np.stack([Lam / (2 * p) for p in tree.prob])
    beta, uh, e = cu.beta @ (f.L.T @ L), cu.u_hat, cu.e

    def step(w, Km, Lm, full):
        s, r = w[:, :nx].copy(), w[:, nx:] @ Km[nx:]
        if full:
            r = r + beta
        for m in range(n - 1, -1, -1):
            r[m] += s[m] @ Km[:nx]
            if m:
                s[tree.parent[m]] += s[m]
                r[tree.parent[m]] += r[m]
        v = np.einsum("nij,nj->ni", Lm, r)
        x = np.zeros((n, nx))
        for m in range(n):
            up = tree.parent[m]
            if m:
                v[m] += v[up]
            x[m] = (x[up] if m else (P["p"] if full else 0)) + Km[:nx] @ v[m] + (e[m] if full else 0)
        return x, v @ Km[nx:].T + (uh if full else 0)

    c = P["cost"]
    ls, lz, lu = _f32(steps["s"])[:, None], _f32(steps["z"])[:, None], _f32(steps["p"])
    mu, gd = _f32(tree.prob * c["W_x"])[:, None], float(np.float32(c["gamma_d"]))
    xs, lo, hi, ul, uh_ = (_f32(c[k]) for k in ("x_s", "x_min", "x_max", "u_min", "u_max"))
    y = [np.zeros((n, nx)), np.zeros((n, nx)), np.zeros((n, L.shape[0]))]
    old, t0, t1 = y, 1.0, 1.0

    def cap(q, most):
        d = np.sqrt((q * q).sum(1, keepdims=True))
        return np.where(d > most, q * (most / np.maximum(d, 1e-300)), q)

    for k in range(iters):
        ex = float(np.float32(t1 * (1 / t0 - 1)))
        w = [a + ex * (a - b) for a, b in zip(y, old)]
        W = np.concatenate([w[0] + w[1], w[2]], axis=1)
        if k % every == 0 or k >= iters - polish:
            Wa = _f32(W)
            x, u = xa, ua = step(Wa, K, L64, True)
        else:
            x, u = step(W - Wa, K16, L16, False)
            x, u = x + xa, u + ua
        ql, qh = w[1] + lz * (x - lo), w[1] + lz * (x - hi)
        pl, ph = w[2] + lu * (u - ul), w[2] + lu * (u - uh_)
        old, y = y, [cap(np.minimum(w[0] + ls * (x - xs), 0), mu),
                     cap(np.where(qh > 0, qh, np.where(ql < 0, ql, 0.0)), gd),
                     np.where(ph > 0, ph, np.where(pl < 0, pl, 0.0))]
        t0, t1 = t1, 0.5 * (math.sqrt(t1 ** 4 + 4 * t1 ** 2) - t1 ** 2)
    return x


@pytest.mark.parametrize("n_x,n_u,n_e,N,every,polish", [(7, 13, 2, 6, 16, 0), (7, 13, 2, 12, 16, 0), (7, 13, 2, 18, 16, 0),
                                                        (20, 40, 6, 6, 16, 0), (20, 40, 6, 12, 16, 0),
                                                        (20, 40, 6, 18, 16, 0), (20, 40, 6, 18, 5, 10),
                                                        (50, 90, 14, 18, 16, 0), (63, 114, 17, 12, 16, 0),
                                                        (63, 114, 17, 18, 16, 0), (63, 114, 17, 18, 5, 10)])
def test_rounding_errors_are_those_of_the_other_schedules(n_x, n_u, n_e, N, every, polish):
    """The two-launch form's distance to the float64 iteration (root mean square of x) is at most
    twice the largest of schedules 1 to 4's, which differ among themselves by up to 1.3: where a
    rounding error is the same in all fifteen steps between two anchors, it is 3 to 8 times as far."""
    P = synth.custom(65, n_x, n_u, max(n_e, 3), n_e, synth.make_tree([4, 4], N))
    steps = {k: np.float32(v).astype(np.float64) for k, v in H.full_size_steps(P).items()}
    want = _anchored(P, steps, 60, every, polish)
    off = {}
    for s in (1, 2, 3, 4, 0):
        g = two_launch(P, steps, precision=2) if s == 0 else H.Gpu(P, steps=steps, precision=2, schedule=s)
        try:
            g.smpc.smpc_solve(g.fac, P["p"], P["q"], P["dhat"], P["alpha2"], eps=P["eps"], max_iters=60, sync=1,
                              anchor_every=every, polish_iters=polish, u=g.u, x=g.x, y=g.y)
            off[s] = np.sqrt(((g.arrays()[1] - want) ** 2).mean())
        finally:
            g.close()
    assert off[0] <= 2 * max(off[s] for s in (1, 2, 3, 4)), off


def test_deeper_trees_keep_schedules_1_to_4():
    P = synth.custom(67, 7, 13, 3, 2, synth.make_tree([2, 2], 19))
    _refused(P, H.full_size_steps(P), precision=2)
