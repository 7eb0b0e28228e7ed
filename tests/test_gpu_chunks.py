"""Partner chunks of small problems (up to 32 per item) on the GPU.

Twelve occupied states on a 15^3 box: tc_init gives the occupied-pair stage 12 chunks of one pair.  Eight, the most
that tc_autotune's own candidates go to, leave two pairs to some CTAs and take about twice as long, so the tuner
has to keep the 12.  Where the device has no room for the workspace of that many parts (TC_FAULT=nochunks: as if
so), contexts and batches take at most 8 and compute the same operator.
"""
import numpy as np
import pytest

from conftest import make_setup
from paper_2302_07420_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _case():
    p = synth.tiny_params(31, kmesh=(1, 2, 2), fft=(15,) * 3, ecut=6.0, nbands=3, nocc=3, scale=5.0)
    S = make_setup(p)
    phi, chi = synth.random_orbitals(synth.SEED0 + 930, [S.kpG(k) for k in range(S.Nk)], S.npw_max, S.nbands, perturb=0.1)
    return p, phi, chi, synth.occupations(S.Nk, S.nbands, S.nocc)


def _ctx(p, **kw):
    from paper_2302_07420_gb300.operator import Context
    return Context(p["lattice"], p["kmesh"], p["ecut"], p["fft"], p["nbands"], p["nocc"], p["A"], p["C"], **kw)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 1e-5)])
def test_autotune_times_the_default_counts(prec, tol):
    p, phi, chi, occ = _case()
    d_phi, d_chi = torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda()
    ctx = _ctx(p, precision=prec)
    try:
        r0, l0 = [x.cpu().numpy() for x in ctx.apply(d_phi, d_chi, occ)]
        so, sc = ctx.autotune(d_phi, d_chi, occ)
        r1, l1 = [x.cpu().numpy() for x in ctx.apply(d_phi, d_chi, occ)]
        again = ctx.autotune(d_phi, d_chi, occ)
    finally:
        ctx.close()
    assert so == 12 and 1 <= sc <= 12 and again[0] == 12, (so, sc, again)
    assert np.abs(r1 - r0).max() < tol * np.abs(r0).max() and np.abs(l1 - l0).max() < tol * np.abs(l0).max()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 1e-5)])
def test_fewer_chunks_where_memory_is_short(prec, tol, monkeypatch):
    from paper_2302_07420_gb300.operator import BatchContext
    p, phi, chi, occ = _case()
    d_phi, d_chi = torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda()
    outs = []
    for fault in (None, "nochunks"):
        if fault:
            monkeypatch.setenv("TC_FAULT", fault)
        ctx = _ctx(p, precision=prec)
        batch = BatchContext([p, p], precision=prec)
        try:
            outs += [x.cpu().numpy() for x in ctx.apply(d_phi, d_chi, occ)]
            r, l = batch.apply([d_phi, d_phi], [d_chi, d_chi], [occ, occ])
            for k in range(2):
                outs += [r[k].cpu().numpy(), l[k].cpu().numpy()]
            if fault:
                so, sc = ctx.autotune(d_phi, d_chi, occ)
                assert so <= 8 and sc <= 8, (so, sc)
        finally:
            batch.close()
            ctx.close()
    for k, x in enumerate(outs):
        assert np.abs(x - outs[k % 2]).max() < tol * np.abs(outs[k % 2]).max()
