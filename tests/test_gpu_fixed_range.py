"""The fixed-point transforms of the FP64 pair kernels over the range of FP64: on the compiled supports
(16^3 span 6, 18^3, 24^3) and on the full support of the small boxes (9^3, 12^3, 15^3, 16^3 span 8).

Scalings by powers of two are exact in FP64 arithmetic, and the exponents of every bound follow them, so the
outputs have to scale bit for bit: orbitals by 2^+-540 and 2^+-600 (squares of such values leave FP64's
range), one output band by 2^+-600 among others, the Jastrow amplitude by 2^+-200 (kernel values far outside
the range of FP32).
"""
import numpy as np
import pytest

from conftest import make_setup
from oracle import operator as OP
from paper_2302_07420_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# box, plane-wave cutoff, kernel kind and support
BOXES = {"f9": (9, 2.0, (0, 9)), "f12": (12, 4.0, (0, 12)), "f15": (15, 6.0, (0, 15)), "f16": (16, 9.0, (0, 16)),
         "p16": (16, 6.0, (1, 13)), "p18": (18, 8.0, (1, 17)), "p24": (24, 10.0, (1, 17))}
_CASES = {}


def _case(name):
    if name not in _CASES:
        n, ecut, kind = BOXES[name]
        p = synth.tiny_params(31, kmesh=(1, 1, 2), fft=(n,) * 3, ecut=ecut, nbands=3, nocc=2, scale=5.0)
        S = make_setup(p)
        phi, chi = synth.random_orbitals(synth.SEED0 + 910 + n, [S.kpG(k) for k in range(S.Nk)], S.npw_max, S.nbands,
                                         perturb=0.1)
        occ = synth.occupations(S.Nk, S.nbands, S.nocc)
        occ[:, : S.nocc] = np.array([1.0, 0.6])[None]
        _CASES[name] = (p, S, phi, chi, occ)
    return _CASES[name]


def _run(name, phi, chi, A_scale=1.0, **kw):
    from paper_2302_07420_gb300.operator import Context
    p, S, _, _, occ = _case(name)
    ctx = Context(p["lattice"], p["kmesh"], p["ecut"], p["fft"], p["nbands"], p["nocc"], [a * A_scale for a in p["A"]],
                  p["C"], **kw)
    try:
        assert all(v[:2] == BOXES[name][2] for v in ctx.pair_kernels().values()), ctx.pair_kernels()
        r, l = ctx.apply(torch.from_numpy(phi).cuda(), torch.from_numpy(chi).cuda(), occ)
        return r.cpu().numpy(), l.cpu().numpy()
    finally:
        ctx.close()


@pytest.mark.parametrize("name", sorted(BOXES))
def test_orbitals_by_powers_of_two(name):
    _, S, phi, chi, occ = _case(name)
    r0, l0 = _run(name, phi, chi)
    for ref, out in zip(OP.tc_apply(S, phi, chi, occ), (r0, l0)):
        assert np.abs(out - ref).max() / np.abs(ref).max() < 1e-11
    for e in (-600, -540, 540, 600):
        r, l = _run(name, phi * 2.0 ** e, chi * 2.0 ** -e)
        assert np.array_equal(r, r0 * 2.0 ** e) and np.array_equal(l, l0 * 2.0 ** -e), e


@pytest.mark.parametrize("name", sorted(BOXES))
@pytest.mark.parametrize("e", [-600, 600])
def test_one_output_band_far_from_the_others(name, e):
    _, S, phi, chi, _ = _case(name)
    r0, l0 = _run(name, phi, chi)
    far = phi.copy()
    far[:, S.nocc] *= 2.0 ** e      # unoccupied: an output only
    r, l = _run(name, far, chi)
    r0[:, S.nocc] *= 2.0 ** e
    assert np.array_equal(r, r0) and np.array_equal(l, l0)


@pytest.mark.parametrize("name", ["f15", "p24"])
@pytest.mark.parametrize("terms,power", [(("2bx1", "2bx2"), 1), (("3a2", "3a4", "3b3", "3b4", "3b5", "3b6"), 2)])
def test_jastrow_amplitude_by_powers_of_two(name, terms, power):
    _, S, phi, chi, _ = _case(name)
    mask = sum(1 << OP.TERMS.index(t) for t in terms)
    r0, l0 = _run(name, phi, chi, term_mask=mask)
    assert np.abs(r0).max() > 0
    for e in (-200, 200):
        r, l = _run(name, phi, chi, A_scale=2.0 ** e, term_mask=mask)
        assert np.array_equal(r, r0 * 2.0 ** (power * e)) and np.array_equal(l, l0 * 2.0 ** (power * e)), e


@pytest.mark.parametrize("name", sorted(BOXES))
def test_nan_and_infinity(name):
    """In an unoccupied band: that orbital's outputs only; in a partner: every output."""
    _, S, phi, chi, _ = _case(name)
    r0, _l = _run(name, phi, chi)
    for value in (np.nan, np.inf):
        bad = phi.copy()
        bad[1, 2, 5] = value
        r, _l = _run(name, bad, chi)
        assert not np.isfinite(r[1, 2, : S.npw[1]]).any()
        keep = np.ones(r.shape[:2], dtype=bool)
        keep[1, 2] = False
        assert np.array_equal(r[keep], r0[keep])
        bad = phi.copy()
        bad[0, 1, 3] = value
        r, l = _run(name, bad, chi)
        for k in range(S.Nk):
            assert not np.isfinite(r[k, :, : S.npw[k]]).any() and not np.isfinite(l[k, :, : S.npw[k]]).any()


@pytest.mark.parametrize("name", sorted(BOXES))
@pytest.mark.parametrize("kind", ["plane_waves", "wide_range", "localised"])
def test_uneven_orbitals_against_the_oracle(name, kind):
    """Single plane waves, coefficients over 200 binary orders, and orbitals localised in different places (the
    norms of their factors are far above that of their product): 1e-11 of the parity tests."""
    _, S, phi, chi, occ = _case(name)
    if kind == "plane_waves":
        phi = np.zeros_like(phi)
        for k in range(S.Nk):
            for b in range(S.nbands):
                phi[k, b, (7 * b + k) % S.npw[k]] = 1.0
        chi = phi.copy()
    elif kind == "wide_range":
        scale = 2.0 ** -np.random.default_rng(7).integers(0, 200, size=phi.shape)
        phi, chi = phi * scale, chi * scale
        phi[:, :, 0] += 1.0
        chi[:, :, 0] += 1.0
    else:
        at = np.array([[0.0, 0.0, 0.0], [0.5, 0.5, 0.5], [0.5, 0.0, 0.5]])   # fractional, one per band
        phi = np.zeros_like(phi)
        for k in range(S.Nk):
            m = np.asarray(S.miller[k])
            for b in range(S.nbands):
                phi[k, b, : len(m)] = np.exp(-0.1 * (m ** 2).sum(1) - 2j * np.pi * (m @ at[b]))
        chi = phi.copy()
    r, l = _run(name, phi, chi)
    for ref, out in zip(OP.tc_apply(S, phi, chi, occ), (r, l)):
        assert np.abs(out - ref).max() / np.abs(ref).max() < 1e-11
