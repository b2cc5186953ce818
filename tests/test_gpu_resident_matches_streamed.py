"""Submatrices of up to 192 rows through both sign kernels, on the same prepared inputs: with the operands on the SM
(nolsm_solve_batch) and streamed (nolsm_sign_noalloc). Single-term products have to keep the streamed kernel's order X T:
T X is as accurate but rounds differently, 2.6e-5 of D away in FP16 (and 2e-4 in BF16). With the same order only single
roundings of the iterates differ, where FP32 sums taken in another order fall on either side: D's relative difference in
the Frobenius norm stays below a fifth of that, 5e-6; the three-term modes round at 2^-22 (BF16X3 after its refinement)."""
import ctypes

import numpy as np
import pytest

from oracle import nolsm_oracle as orc
from synth import SystemSpec, make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp16", "bf16", "fp32", "bf16x3"])
def test_resident_matches_streamed(prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08245_gb300 import build
    build.build()
    import paper_2104_08245_gb300 as nl
    lib = nl._abi.load()
    sysm = make_system(SystemSpec(6, 5, 4, density_amp=0.15, seed=21))
    po = orc.build_plan(sysm.nbf, sysm.S.row_ptr, sysm.S.col_idx, sysm.H.row_ptr, sysm.H.col_idx)
    sel = [J for J in range(sysm.n_mol) if po.sub_n[J] <= 192]
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
    opts = nl.options(prec)
    mu = -0.1
    nl.nolsm_solve_batch(plan, mu, opts, check=False)
    D = plan.scatter().cpu().numpy()
    A, Q, _, _ = nl.nolsm_plan_get_prepared(plan, opts)
    n, b = po.sub_n.astype(np.int64), po.nbf.astype(np.int64)
    a_off, c_off = np.concatenate([[0], np.cumsum(n * n)]), np.concatenate([[0], np.cumsum(n * b)])
    Sc, Hc = np.zeros(c_off[-1]), np.zeros(c_off[-1])
    for J in sel:
        for out, M in ((Sc, sysm.S), (Hc, sysm.H)):
            c0 = int(po.sub_c0[J])
            out[c_off[J]:c_off[J + 1]] = orc.gather(po, J, M.row_ptr, M.col_idx, M.blk_off, M.vals)[:, c0:c0 + b[J]].ravel()
    T = lambda x, dt: torch.as_tensor(np.ascontiguousarray(x), dtype=dt).cuda()
    sub_n, nbf, ao, co = T(n[sel], torch.int32), T(b[sel], torch.int32), T(a_off[sel], torch.int64), T(c_off[sel], torch.int64)
    Scd, Hcd = T(Sc, torch.float64), T(Hc, torch.float64)
    lamd = T(nl.nolsm_features(plan, mu, opts).cpu().numpy()[sel, 1:3].astype(np.float64).ravel(), torch.float64)   # Gershgorin
    Dc = torch.zeros(int(c_off[-1]), dtype=torch.float64, device="cuda")
    tS, tH = (torch.zeros(len(sel), dtype=torch.float64, device="cuda") for _ in range(2))
    it, st = (torch.zeros(len(sel), dtype=torch.int32, device="cuda") for _ in range(2))
    rc = lib.nolsm_sign_noalloc(len(sel), sub_n.data_ptr(), nbf.data_ptr(), ao.data_ptr(), co.data_ptr(), A.data_ptr(),
                                Q.data_ptr(), Scd.data_ptr(), Hcd.data_ptr(), lamd.data_ptr(), mu, ctypes.byref(opts),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), Dc.data_ptr(), tS.data_ptr(),
                                tH.data_ptr(), it.data_ptr(), st.data_ptr())
    assert rc == 0, lib.nolsm_last_error().decode()
    torch.cuda.synchronize()
    assert np.all(st.cpu().numpy() == 0)
    Dc = Dc.cpu().numpy()
    off = orc.d_block_offsets(po)
    diff = norm = 0.0
    for J in sel:
        cols = Dc[c_off[J]:c_off[J + 1]].reshape(n[J], b[J])
        for p in range(po.nb_ptr[J], po.nb_ptr[J + 1]):
            I = int(po.nb_idx[p])
            q = po.nb_ptr[I] + int(np.nonzero(po.nb_idx[po.nb_ptr[I]:po.nb_ptr[I + 1]] == J)[0][0])
            got = D[off[q]:off[q + 1]].reshape(b[I], b[J])
            want = cols[po.nb_off[p]:po.nb_off[p] + b[I]]
            diff += float(np.sum((got - want) ** 2))
            norm += float(np.sum(want ** 2))
    print(f"{prec}: {len(sel)} submatrices, relative difference {np.sqrt(diff / norm):.2e}")
    assert np.sqrt(diff / norm) <= 5e-6
