"""The power iteration and the network's training step at the edges of their kernels' sizes.

Power bounds: fully connected clusters of exactly n rows (four rows a warp, 128 columns a pass, up to 32 warps), against
the FP64 iteration of the oracle. 30 normalised FP32 products leave at most some 2^-24 sqrt(n) of the Gershgorin interval,
which the extrapolation by 5 % of the width passes on: 1e-4 of the width as in the other test, and 1e-6 of the interval
where the width is nothing (n = 1).

Training: a minibatch drawn by index and one launch for the gradients' sum and Adam, against the gradient of the gathered
batch and a separate Adam step; the same arithmetic, so that only the contraction of single roundings may differ."""
import numpy as np
import pytest

from oracle import bounds_oracle as bo
from test_gpu_tile_edges import clusters, lattice_pair

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 3, 4, 5, 31, 33, 127, 128, 129, 161, 255, 257, 530)


@pytest.fixture(scope="module")
def nl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08245_gb300 import build
    build.build()
    import paper_2104_08245_gb300 as nl
    return nl


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_power_bounds_at_the_edges(nl, prec):
    sysm, _ = clusters(SIZES, lattice_pair, 0.5)
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
    o = nl.options(prec)
    lam = nl.nolsm_power_bounds(plan, o).cpu().numpy()
    f = nl.nolsm_features(plan, -0.1, o).cpu().numpy()
    J, p = 0, 0
    for n in SIZES:
        w = 0
        while sum(sysm.nbf[J:J + w]) < n:
            w += 1
        # the cluster's dense pair from its blocks, row by row
        def dense(M):
            out, q = np.zeros((n, n)), p
            off = np.concatenate([[0], np.cumsum(sysm.nbf[J:J + w])])
            for i in range(w):
                for j in range(w):
                    out[off[i]:off[i + 1], off[j]:off[j + 1]] = M.vals[M.blk_off[q]:M.blk_off[q + 1]].reshape(
                        sysm.nbf[J + i], sysm.nbf[J + j])
                    q += 1
            return out
        A = np.linalg.solve(dense(sysm.S), dense(sysm.H))
        lo, hi = float(f[J, 1]), float(f[J, 2])
        ref = bo.power_bounds(A, lo, hi, iters=30)
        tol = 1e-4 * (ref[1] - ref[0]) + 1e-6 * max(hi - lo, 1.0)
        for k in range(w):
            assert abs(lam[J + k, 0] - ref[0]) <= tol and abs(lam[J + k, 1] - ref[1]) <= tol, (n, k, lam[J + k], ref)
        J += w
        p += w * w


@pytest.mark.parametrize("N,batch", [(1, 4), (31, 32), (33, 33), (100, 32), (2600, 1300)])
def test_training_is_gradients_and_adam(nl, N, batch):
    import torch
    rng = np.random.default_rng(N)
    x = torch.from_numpy(rng.normal(size=(N, 7)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(size=(N, 3)).astype(np.float32)).cuda()
    a, b = nl.Mlp(seed=3), nl.Mlp(seed=3)
    a.train(x, t, 2, batch, 1e-3)
    bs = min(batch, N)
    for e in range(2):
        for start in range(0, N, bs):
            idx = (np.arange(start, min(start + bs, N)) * 7919 + e * 104729) % N
            i = torch.from_numpy(idx).cuda()
            b.gradient(x[i].contiguous(), t[i].contiguous())
            b.adam_step(1e-3)
    assert float(np.max(np.abs(a.get_params() - b.get_params()))) <= 1e-6
