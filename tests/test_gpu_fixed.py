"""The fixed-point transforms of the FP64 pruned kernels, where their scaling can go wrong.

Powers of two in the orbitals must pass through bit for bit (the exponents of every bound shift with
them); a NaN in an output orbital must make that orbital's outputs NaN and leave the others alone
(partners: every output); orbitals that are single plane waves (spectra with one nonzero value), with a very small
occupied weight, and with coefficients spread over 200 binary orders keep the 1e-11 of the parity tests
against the FP64 oracle.
"""
import numpy as np
import pytest

from conftest import make_setup
from oracle import operator as OP
from paper_2302_07420_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CELLS = {
    "n16": lambda: synth.tiny_params(31, kmesh=(1, 1, 2), fft=(16,) * 3, ecut=6.0, nbands=3, nocc=2, scale=5.0),
    "n20": lambda: synth.tiny_params(33, kmesh=(1, 2, 1), fft=(20,) * 3, ecut=10.0, nbands=3, nocc=2, scale=5.0),
    "n24": lambda: synth.si_params(kmesh=(1, 1, 2), nbands=3, nocc=2),
}


def _case(name):
    from paper_2302_07420_gb300.operator import Context
    p = CELLS[name]()
    S = make_setup(p)
    phi, chi = synth.random_orbitals(synth.SEED0 + 900 + S.n[0], [S.kpG(k) for k in range(S.Nk)], S.npw_max, S.nbands,
                                     perturb=0.1)
    occ = synth.occupations(S.Nk, S.nbands, S.nocc)
    occ[:, : S.nocc] = np.array([1.0, 0.6])[None]
    ctx = Context(p["lattice"], p["kmesh"], p["ecut"], p["fft"], p["nbands"], p["nocc"], p["A"], p["C"])
    assert all(v[0] == 1 for v in ctx.pair_kernels().values())
    return S, phi, chi, occ, ctx


def _run(ctx, phi, chi, occ):
    r, l = ctx.apply(torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda(), occ)
    return r.cpu().numpy(), l.cpu().numpy()


def _close(S, phi, chi, occ, got):
    for ref, out in zip(OP.tc_apply(S, phi, chi, occ), got):
        assert np.abs(out - ref).max() / np.abs(ref).max() < 1e-11


@pytest.mark.parametrize("name", sorted(CELLS))
def test_powers_of_two_pass_through(name):
    S, phi, chi, occ, ctx = _case(name)
    r0, l0 = _run(ctx, phi, chi, occ)
    for e in (-150, -3, 200):
        r, l = _run(ctx, phi * 2.0 ** e, chi * 2.0 ** -e, occ)
        assert np.array_equal(r, r0 * 2.0 ** e) and np.array_equal(l, l0 * 2.0 ** -e)


def test_nan_stays_where_it_belongs():
    S, phi, chi, occ, ctx = _case("n24")
    r0, _ = _run(ctx, phi, chi, occ)
    bad = phi.copy()
    bad[1, 2, 5] = np.nan       # an unoccupied band: an output only
    r, _ = _run(ctx, bad, chi, occ)
    assert np.isnan(r[1, 2, : S.npw[1]]).all()
    keep = np.ones(r.shape[:2], dtype=bool)
    keep[1, 2] = False
    assert np.array_equal(r[keep], r0[keep])
    bad = phi.copy()
    bad[0, 1, 3] = np.inf       # a partner: every output
    r, l = _run(ctx, bad, chi, occ)
    for k in range(S.Nk):
        assert not np.isfinite(r[k, :, : S.npw[k]]).any() and not np.isfinite(l[k, :, : S.npw[k]]).any()


@pytest.mark.parametrize("kind", ["plane_waves", "tiny_weight", "wide_range"])
def test_uneven_orbitals_against_the_oracle(kind):
    S, phi, chi, occ, ctx = _case("n24")
    if kind == "plane_waves":
        phi = np.zeros_like(phi)
        for k in range(S.Nk):
            for b in range(S.nbands):
                phi[k, b, 7 * b + k] = 1.0
        chi = phi.copy()
    elif kind == "tiny_weight":
        occ[0, 1] = 1e-30
        occ[1, 0] = 1e-9
    else:
        rng = np.random.default_rng(7)
        scale = 2.0 ** -rng.integers(0, 200, size=phi.shape)
        phi, chi = phi * scale, chi * scale
        phi[:, :, 0] += 1.0
        chi[:, :, 0] += 1.0
    _close(S, phi, chi, occ, _run(ctx, phi, chi, occ))
