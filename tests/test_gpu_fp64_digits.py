"""The FP64 class's exact digit products (two CTAs a submatrix): the course of a cluster, and overlaps of every condition.

Reference: the eigenvectors of (H, S) below mu, in FP64."""
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
