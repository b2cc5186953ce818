"""The centre columns of T_J(S)^-1 after the tensor-core inverse, on overlaps between well and ill conditioned.

Pairs of functions that overlap by +-s have S_ii (S^-1)_ii = 1 / (1 - s^2), the estimate that the modes accept up to 10
(FP32) or 30; the products S_ik (S^-1)_kc that the residual adds up reach it, and cancel. The refinement stops after a
correction below 1e-5 of q, whose square is left: within 1e-10 of the largest entry."""
import types

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ESTIMATES = (1.1, 3.0, 5.0, 8.0, 10.0, 25.0)
WIDTHS = {168: 6, 192: 8, 264: 6, 46: 23}      # rows of a submatrix: functions a molecule


@pytest.fixture(scope="module")
def nl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08245_gb300 import build
    build.build()
    import paper_2104_08245_gb300 as nl
    return nl


def overlap(n, est, rng):
    """Pairs at random places with either sign, and a weak coupling between all functions."""
    E = rng.normal(size=(n, n))
    S = np.eye(n) + 0.002 * (E + E.T) / np.sqrt(n)
    np.fill_diagonal(S, 1.0)
    p = rng.permutation(n)
    s = np.sqrt(1.0 - 1.0 / est) * np.where(rng.random(n // 2) < 0.5, 1.0, -1.0)
    S[p[0:2 * (n // 2):2], p[1::2]] = S[p[1::2], p[0:2 * (n // 2):2]] = s
    return S


@pytest.mark.parametrize("n,est", [(n, e) for n in WIDTHS for e in ESTIMATES])
def test_centre_columns(nl, n, est):
    rng = np.random.default_rng(int(1000 * est) + n)
    b = WIDTHS[n]
    m = n // b
    S = overlap(n, est, rng)
    H = np.diag(np.resize([-1.0, -0.5, 0.3], n))
    blocks = lambda M: np.concatenate([M[b * i:b * i + b, b * j:b * j + b].ravel() for i in range(m) for j in range(m)])  # noqa: E731
    csr = lambda M: types.SimpleNamespace(row_ptr=np.arange(0, m * m + 1, m), col_idx=np.tile(np.arange(m), m), vals=blocks(M))  # noqa: E731
    sysm = types.SimpleNamespace(nbf=np.full(m, b), S=csr(S), H=csr(H), n_occ=1.0)
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
    _, Q, status, cond = nl.nolsm_plan_get_prepared(plan, nl.options("bf16x3", inverse=1))
    assert np.all(status.cpu().numpy() == 0)
    exact = np.linalg.inv(S)
    Q = Q.cpu().numpy().reshape(m, n, b)
    err = max(float(np.max(np.abs(Q[J] - exact[:, b * J:b * J + b]))) for J in range(m)) / float(np.max(np.abs(exact)))
    print(f"n {n}, estimate {float(cond.max()):.2f}: relative max|dQ| = {err:.2e}")
    assert err <= 1e-10
    plan.close()
