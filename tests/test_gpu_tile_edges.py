"""Submatrices whose dimension sits on the edges of the kernels' tiles, in every precision class.

One system holds a fully connected cluster of molecules per dimension n, so that each of its submatrices has exactly n
rows: 1 row, the edges of the 16-row K steps, of the 32-column chunks, 64-column blocks and 128-row tiles, 192 and 193
(operands kept on the SM or streamed), 512 and 513 (digits of 9 or 8 bits in the FP64 products). The functions per
molecule run from 1 to 13, past the eight columns that one pass of the centre-column kernels takes. Reference: the
eigenvectors of (H, S) below mu, in FP64.

FP64: dense random S = I + E, |E|_2 = spread, which sets the steps of the inverse square root (0.0005: one, 0.1: two,
0.6: more, each another route), and levels in [-1, -0.5] and [0.3, 0.8]; within 1e-10, as an iteration that ends with a
quadratic step below 1e-9 leaves nothing above its rounding. FP32, BF16X3 and FP16: clusters of the kind that the
precision targets are stated for (Gaussian overlaps over a jittered lattice), at those targets; the Gaussian's exponent
sets the steps of the inverse square root in the same way."""
import types

import numpy as np
import pytest
import scipy.linalg

from oracle import nolsm_oracle as orc

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 15, 16, 17, 31, 33, 63, 64, 65, 95, 127, 128, 129, 159, 160, 161, 176, 191, 192, 193, 257)
SIZES_FP64 = SIZES + (511, 512, 513, 530)
TOL = {"fp64": 1e-10, "fp32": 1e-6, "bf16x3": 1e-4, "fp16": 1e-4}
MU = -0.1


@pytest.fixture(scope="module")
def nl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08245_gb300 import build
    build.build()
    import paper_2104_08245_gb300 as nl
    return nl


def random_pair(w, spread, rng):
    n = sum(w)
    E = rng.normal(size=(n, n))
    s, V = np.linalg.eigh(np.eye(n) + spread * (E + E.T) / np.linalg.norm(E + E.T, 2))
    U = np.linalg.qr(rng.normal(size=(n, n)))[0]
    m = (2 * n + 2) // 3
    eps = np.concatenate([rng.uniform(-1.0, -0.5, m), rng.uniform(0.3, 0.8, n - m)])
    root = (V * np.sqrt(s)) @ V.T
    return (V * s) @ V.T, root @ (U * eps) @ U.T @ root


def lattice_pair(w, s_exp, rng):
    k = int(np.ceil(len(w) ** (1 / 3) - 1e-9))
    pos = 3.1 * np.array([(i % k, i // k % k, i // (k * k)) for i in range(len(w))]) + rng.uniform(-0.3, 0.3, (len(w), 3))
    of = np.repeat(np.arange(len(w)), w)
    r = np.linalg.norm(pos[of][:, None] - pos[of][None], axis=2)
    scale = 1.0 / np.sqrt(np.outer(np.array(w)[of], np.array(w)[of]))
    other = of[:, None] != of[None]
    level = np.concatenate([np.resize([-1.0, -0.5, -0.5, -0.5, 0.3, 0.3], b) for b in w])
    return (np.where(other, scale * np.exp(-s_exp * r * r), np.eye(len(of))),
            np.where(other, -0.2 * scale * np.exp(-r / 1.5), np.diag(level)))


def clusters(sizes, pair, arg, seed=5):
    """(system, exact density per cluster)"""
    rng = np.random.default_rng(seed)
    nbf, row_ptr, cols, blocks, exact, occ = [], [0], [], {"S": [], "H": []}, [], 0
    for n in sizes:
        w = []
        while sum(w) < n:
            w.append(min((6, 1, 8, 13, 3)[len(w) % 5], n - sum(w)))
        M = dict(zip("SH", (0.5 * (m + m.T) for m in pair(w, arg, rng))))
        eps, C = scipy.linalg.eigh(M["H"], M["S"])
        assert np.min(np.abs(eps - MU)) > 0.1
        C = C[:, eps < MU]
        exact.append(C @ C.T)
        occ += C.shape[1]
        first, off = len(nbf), np.concatenate([[0], np.cumsum(w)])
        for i in range(len(w)):
            cols.extend(range(first, first + len(w)))
            row_ptr.append(len(cols))
            for k in M:
                blocks[k].extend(M[k][off[i]:off[i + 1], off[j]:off[j + 1]].ravel() for j in range(len(w)))
        nbf.extend(w)

    def csr(k):
        return types.SimpleNamespace(row_ptr=np.array(row_ptr, np.int32), col_idx=np.array(cols, np.int32),
                                     blk_off=np.concatenate([[0], np.cumsum([x.size for x in blocks[k]])]),
                                     vals=np.concatenate(blocks[k]))
    return types.SimpleNamespace(nbf=np.array(nbf, np.int32), S=csr("S"), H=csr("H"), n_occ=float(occ)), exact


def solved(nl, prec, sizes, pair, arg):
    sysm, exact = clusters(sizes, pair, arg)
    po = orc.build_plan(sysm.nbf, sysm.S.row_ptr, sysm.S.col_idx, sysm.H.row_ptr, sysm.H.col_idx)
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
    r = nl.nolsm_solve_batch(plan, MU, nl.options(prec))
    assert np.all(r.sub_status.cpu().numpy() == 0)
    D = orc.d_to_dense(po, plan.scatter().cpu().numpy())
    at, err = 0, {}
    for n, ref in zip(sizes, exact):
        err[n] = float(np.max(np.abs(D[at:at + n, at:at + n] - ref)))
        at += n
    print(f"{prec}, {arg}: max|dD| = {max(err.values()):.3e}")
    assert max(err.values()) <= TOL[prec], err


@pytest.mark.parametrize("prec,arg", [(p, a) for p in TOL for a in ((0.0005, 0.1, 0.6) if p == "fp64" else (1.2, 0.5, 0.25))])
def test_every_tile_edge(nl, prec, arg):
    sizes = SIZES_FP64 if prec == "fp64" else SIZES
    solved(nl, prec, sizes, random_pair if prec == "fp64" else lattice_pair, arg)


@pytest.mark.parametrize("sizes", [(193, 255, 257), (321, 384, 385, 512), (448, 513, 640, 767, 961)])
def test_groups_of_ctas(nl, sizes):
    """Streamed submatrices shared by two, four and eight CTAs (by their mean dimension), with one to four column tiles,
    and a Q of more rows than one staged piece."""
    solved(nl, "bf16x3", sizes, lattice_pair, 0.5)
