"""The FP64 class's exact digit products (two CTAs a submatrix): the course of a cluster, and overlaps of every condition.

Reference: the eigenvectors of (H, S) below mu, in FP64."""
import types

import numpy as np
import pytest

from oracle import nolsm_oracle as orc
from test_gpu_tile_edges import MU, clusters, random_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08245_gb300 import build
    build.build()
    import paper_2104_08245_gb300 as nl
    return nl


def test_submatrices_without_a_tile_for_the_second_cta_and_starts_that_give_up(nl):
    """Several submatrices a cluster of 1 to 64 rows, of which the second CTA of a cluster has no tile, and every third
    pair scaled by 1e-7, whose inverse lies outside the digits' range: its preparation gives up at the start and leaves
    it to the FP64 factorisation, with the next one following at once. Every role has to keep to the meetings then.
    Within 1e-10 of the largest entry, as an iteration that ends with a quadratic step below 1e-9 leaves nothing above
    its rounding."""
    rng = np.random.default_rng(11)
    sizes = [int(n) for n in rng.integers(1, 41, 300)] + [64, 63, 1, 17] * 5
    made = iter(range(len(sizes)))

    def pair(w, spread, rng):
        S, H = random_pair(w, spread, rng)
        c = 1e-7 if next(made) % 3 == 0 else 1.0
        return c * S, c * H

    sysm, exact = clusters(sizes, pair, 0.1)
    po = orc.build_plan(sysm.nbf, sysm.S.row_ptr, sysm.S.col_idx, sysm.H.row_ptr, sysm.H.col_idx)
    for _ in range(3):
        plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
        r = nl.nolsm_solve_batch(plan, MU, nl.options("fp64"))
        assert np.all(r.sub_status.cpu().numpy() == 0)
        D = orc.d_to_dense(po, plan.scatter().cpu().numpy())
        at, err = 0, 0.0
        for n, ref in zip(sizes, exact):
            err = max(err, float(np.max(np.abs(D[at:at + n, at:at + n] - ref)) / max(1.0, np.max(np.abs(ref)))))
            at += n
        print(f"{len(sizes)} clusters: relative max|dD| = {err:.3e}")
        assert err <= 1e-10
        plan.close()


def conditioned(kind, n, cond, rng):
    """(S, H) in FP64 with eigenvalues of S spread over cond: one small one, logarithmically, or 1 +- s in pairs."""
    if kind == "pairs":
        p, S = rng.permutation(n), np.eye(n)
        E = rng.normal(size=(n, n))
        S[p[0::2], p[1::2]] = S[p[1::2], p[0::2]] = (cond - 1) / (cond + 1) * np.where(rng.random(n // 2) < 0.5, 1.0, -1.0)
        S += 1e-4 * (E + E.T) / np.sqrt(n) * min(1.0, 10.0 / cond)
    else:
        s = np.exp(np.linspace(0.0, -np.log(cond), n)) if kind == "log" else rng.uniform(1.0, 1.2, n)
        if kind == "one":
            s[0] = 1.1 / cond
        V = np.linalg.qr(rng.normal(size=(n, n)))[0]
        S = (V * s) @ V.T
    s, V = np.linalg.eigh(0.5 * (S + S.T))
    root = (V * np.sqrt(s)) @ V.T
    U = np.linalg.qr(rng.normal(size=(n, n)))[0]
    eps = np.concatenate([rng.uniform(-1.0, -0.5, 2 * n // 3), rng.uniform(0.3, 0.8, n - 2 * n // 3)])
    H = root @ (U * eps) @ U.T @ root
    return 0.5 * (S + S.T), 0.5 * (H + H.T)


def extended(S, H):
    """T_J(S)^-1, A and the density of (S, H) in numpy's extended precision (80 or 128 bits)."""
    I = np.eye(len(S), dtype=np.longdouble)
    X, Sl = np.linalg.inv(S).astype(np.longdouble), S.astype(np.longdouble)
    for _ in range(2):
        X = X + X @ (I - Sl @ X)
    A = X @ H.astype(np.longdouble)
    W = A - np.longdouble(MU) * I
    W = W / np.max(np.sum(np.abs(W), axis=1))
    for _ in range(60):
        P = W @ W
        W = (3 * W - W @ P) / 2
        if float(np.max(np.abs(I - P))) < 1e-9:
            break
    return X, A, (X - W @ X) / 2


@pytest.mark.parametrize("kind", ["one", "log", "pairs"])
@pytest.mark.parametrize("cond", [2, 10, 50, 250, 1000])
def test_as_accurate_as_fp64_arithmetic_on_every_overlap(nl, kind, cond):
    """A_J, the centre columns of T_J(S)^-1 and the density against extended precision. A Cholesky factorisation and
    its solves in FP64 leave some cond x 2^-53 of the largest entry; three times that, and 2e-15 for the sums of 60 terms."""
    n, b = 60, 6
    m = n // b
    S, H = conditioned(kind, n, cond, np.random.default_rng(cond + 7))
    ref = extended(S, H)
    blocks = lambda M: np.concatenate([M[b * i:b * i + b, b * j:b * j + b].ravel() for i in range(m) for j in range(m)])  # noqa: E731
    csr = lambda M: types.SimpleNamespace(row_ptr=np.arange(0, m * m + 1, m), col_idx=np.tile(np.arange(m), m), vals=blocks(M))  # noqa: E731
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(types.SimpleNamespace(nbf=np.full(m, b), S=csr(S), H=csr(H), n_occ=1.0)))
    nl.nolsm_solve_batch(plan, MU, nl.options("fp16", inverse=1), check=False)   # a tensor-core mode's hand-over comes first
    o = nl.options("fp64")
    A, Q, _, _ = nl.nolsm_plan_get_prepared(plan, o)
    r = nl.nolsm_solve_batch(plan, MU, o)
    D = plan.scatter().cpu().numpy().reshape(m, m, b, b).transpose(0, 2, 1, 3).reshape(n, n)
    got = (np.concatenate(list(Q.cpu().numpy().reshape(m, n, b)), axis=1), A.cpu().numpy()[:n * n].reshape(n, n), D)
    err = [float(np.max(np.abs(g - e)) / np.max(np.abs(e))) for g, e in zip(got, ref)]
    print(f"{kind}, condition {cond}: Q {err[0]:.1e}, A {err[1]:.1e}, D {err[2]:.1e}, {int(r.iters[0])} steps")
    assert max(err) <= 2e-15 + 3.0 * cond * 2.0 ** -53
    plan.close()


def test_without_room_for_the_digit_planes_the_fp64_kernels_take_over(nl):
    """20 submatrices of 600 rows need some 0.4 GB with the FP64 kernels and 1 GB with the digit products; 0.52 GB are
    left free. The density is that of a solve with room, to 1e-12."""
    import ctypes

    import torch
    n, b = 600, 30
    m = n // b
    S, H = conditioned("log", n, 2, np.random.default_rng(3))
    blocks = lambda M: np.concatenate([M[b * i:b * i + b, b * j:b * j + b].ravel() for i in range(m) for j in range(m)])  # noqa: E731
    csr = lambda M: types.SimpleNamespace(row_ptr=np.arange(0, m * m + 1, m), col_idx=np.tile(np.arange(m), m), vals=blocks(M))  # noqa: E731
    dsys = nl.DeviceSystem(types.SimpleNamespace(nbf=np.full(m, b), S=csr(S), H=csr(H), n_occ=1.0))

    def solve():
        plan = nl.nolsm_build_submatrices(dsys)
        r = nl.nolsm_solve_batch(plan, MU, nl.options("fp64"))
        assert np.all(r.sub_status.cpu().numpy() == 0)
        D, used = plan.scatter().cpu().numpy(), plan.info().device_bytes
        plan.close()
        return D, used

    D0, used0 = solve()
    cuda, pool = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert cuda.cuMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    filled = torch.empty(torch.cuda.mem_get_info()[0] - 520 * 2 ** 20, dtype=torch.uint8, device="cuda")
    try:
        D1, used1 = solve()
    finally:
        del filled
        torch.cuda.empty_cache()
    print(f"{used0 / 2 ** 20:.0f} MB with room, {used1 / 2 ** 20:.0f} without; max|dD| = {np.max(np.abs(D1 - D0)):.1e}")
    assert used1 < 520 * 2 ** 20 < used0
    assert np.max(np.abs(D1 - D0)) <= 1e-12 * np.max(np.abs(D0))
