"""Launch routes of the pipeline that other cases do not take, against the oracle.

* A Davidson step on 25^3: its second operator launch computes the new vectors' outputs only (output items that
  start after the partners), on the cluster kernels.
* One orbital on boxes whose volume does not fit shared memory (FP64 25^3, FP32 48^3): the scratch holds fewer work
  volumes than the merged Hartree-type launch has, so its kinds run one at a time.
"""
import numpy as np
import pytest

from conftest import make_setup
from oracle import davidson as DV
from oracle import operator as OP
from paper_2302_07420_gb300 import synth

from test_gpu_davidson import _case, _compare, _ctx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,tol_eig,tol_vec", [("fp64", 1e-11, 1e-9), ("fp32", 2e-6, 2e-4)])
def test_davidson_step_on_clusters(prec, tol_eig, tol_vec):
    p, S, phi, chi, occ = _case(8, (1, 1, 2), (25, 25, 25), 4.0, 3, 2)
    ref = DV.davidson_step(S, phi, chi, occ)
    ctx = _ctx(p, precision=prec)
    try:
        assert ctx.pair_kernels()["pair_chain"][0] == 2
        phi_g, chi_g, eig, dim = ctx.davidson_step(torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda(), occ)
        got = (phi_g.cpu().numpy(), chi_g.cpu().numpy(), eig, dim)
    finally:
        ctx.close()
    _compare(S, ref, got, tol_eig, tol_vec)


@pytest.mark.parametrize("prec,n,tol", [("fp64", 25, 1e-11), ("fp32", 48, 1e-5)])
def test_one_orbital_beyond_shared_memory(prec, n, tol):
    p = synth.tiny_params(9, kmesh=(1, 1, 1), fft=(n,) * 3, ecut=2.0, nbands=1, nocc=1, scale=5.0)
    S = make_setup(p)
    phi, chi = synth.random_orbitals(synth.SEED0 + 940 + n, [S.kpG(0)], S.npw_max, 1, perturb=0.1)
    occ = np.ones((1, 1))
    ctx = _ctx(p, precision=prec)
    try:
        ctx.profile(True)
        r, l = ctx.apply(torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda(), occ)
        assert ctx.stage_times()["hartree"][1] == 8      # five launches where the merged one fits
        r, l = r.cpu().numpy(), l.cpu().numpy()
    finally:
        ctx.close()
    for ref, out in zip(OP.tc_apply(S, phi, chi, occ), (r, l)):
        assert np.abs(out - ref).max() / np.abs(ref).max() < tol
