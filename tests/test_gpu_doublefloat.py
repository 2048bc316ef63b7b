"""The log det and the gradient of E1 of the mixed path at the precision of their arithmetic (double-float, 48 bits).

Log det: the reference is the FP64 log det of the walker that the call returned, so that nothing of the
22-bit split GEMMs enters.  An error dS of the overlap and its factorisation moves log det S by
tr(S^-1 dS), so the bar is
  u sum_ij |S^-1|_ji (|A^dag| |phi| + P |L| |U|)_ij,  S = P L U.
Each entry of dS gathers up to M products and up to N updates whose roundings are at most 2^-47 of
the terms and about 2^-49 in the mean; they differ in sign from entry to entry, so that the sum
of absolute values over all N^2 entries outweighs their number: u = 2^-48.  The inverse's elimination
(the log det of a step with energies) forms the panels' transforms explicitly, one rounding more per
update: u = 2^-47.

Walkers: near the trial; random (row exchanges in every panel); random with the occupied rows
graded over six decades, where M >= 2 nocc keeps the walker's columns independent (orthonormalise only:
one propagation from there overflows).
"""
import numpy as np
import pytest
import scipy.linalg

import gen
from oracle import afqmc_kp as ok

torch = pytest.importorskip("torch")
from gpu_util import dev, host, make, wrap_phase  # noqa: E402

pytestmark = pytest.mark.gpu


def spec(grid, nocc, M, nw=2):
    return gen.SystemSpec(grid=grid, M=M, nocc=nocc, nchol=2, nwalkers=nw, dt=0.01, seed=1)


# one CTA per matrix with four, two and two lanes per row; two, four and eight CTAs
SIZES = {"N16": ((2, 2, 2), 2, 4), "N27": ((3, 3, 3), 1, 2), "N48": ((2, 2, 3), 4, 8), "N65": ((5, 1, 1), 13, 15),
         "N108": ((3, 3, 3), 4, 8), "N128": ((4, 4, 1), 8, 16), "N120": ((4, 2, 1), 15, 16), "N160": ((4, 4, 1), 10, 11),
         "N256": ((4, 4, 1), 16, 17)}


def walkers(sp, kind):
    """Two walkers."""
    if kind == "near":
        return gen.near_trial_walkers(sp, 2)
    phi = gen.walkers(sp, 2)
    if kind == "graded":   # the trial is the first nocc orbitals of every k: row (k, a) of S is row (k, a) of phi
        grade = 10.0 ** (-6.0 * np.random.default_rng(3).permutation(sp.N) / (sp.N - 1))
        phi.reshape(2, 2, sp.nk, sp.M, sp.N)[:, :, :, :sp.nocc] *= grade.reshape(sp.nk, sp.nocc)[..., None]
    return phi


def calls(sys_, phis, kind):
    """{call: (walkers it returned, their log det)}"""
    sp_w = phis.shape[0]
    x = torch.zeros(sys_.field_shape, dtype=torch.float64, device="cuda")
    out = {}
    for call in ("orthonormalise",) if kind == "graded" else ("orthonormalise", "propagate", "step"):
        phi, w = dev(phis), torch.ones(sp_w, dtype=torch.float64, device="cuda")
        ld = torch.empty((sp_w, 2), dtype=torch.complex128, device="cuda")
        if call == "orthonormalise":
            sys_.orthonormalise(phi, ld)
        elif call == "propagate":
            sys_.propagate(phi, x, w, logdet=ld)
        else:
            sys_.step(phi, x, w, logdet=ld, reuse=False)
        out[call] = host(phi), host(ld)
    return out


def reference(Ad, phi):
    """(log det A^dag phi, the bar's sum)"""
    S = Ad.conj().T @ phi
    P, L, U = scipy.linalg.lu(S)
    terms = np.abs(Ad).T @ np.abs(phi) + P @ (np.abs(L) @ np.abs(U))
    sign, mag = np.linalg.slogdet(S)
    return mag + 1j * np.angle(sign), np.sum(np.abs(np.linalg.inv(S)).T * terms)


CASES = [(name, kind) for name, (_, nocc, M) in SIZES.items() for kind in ("near", "random", "graded")
         if kind != "graded" or M >= 2 * nocc]


@pytest.mark.parametrize("name,kind", CASES)
def test_log_det(name, kind):
    sp = spec(*SIZES[name])
    sys_, osys = make(sp, "mixed")
    Ad = osys.A_dense()
    for call, (phi, ld) in calls(sys_, walkers(sp, kind), kind).items():
        u = 2.0 ** (-47 if call == "step" else -48)
        for w in range(2):
            for s in range(2):
                ref, bar = reference(Ad, phi[w, s])
                d = ld[w, s] - ref
                assert max(abs(d.real), abs(wrap_phase(d.imag))) < u * bar, (call, w, s, d, u * bar)
    assert sys_.last_error() == (0, 0)
    sys_.close()


# both sides of the choice between clusters and the global form, and clusters of different sizes
BATCH = {"N27": 64, "N108": 64, "N120": 152, "N160": 64, "N256": 64}


@pytest.mark.parametrize("name", list(BATCH))
def test_log_det_does_not_depend_on_the_batch(name):
    """A walker's log det has the same bits alone (two walkers) and among many (of the sizes at which the force
    bias, whose k blocks are grouped by the number of tiles, returns the same walkers)."""
    got = []
    for nw in (2, BATCH[name]):
        sp = spec(*SIZES[name], nw=nw)
        sys_, _ = make(sp, "mixed")
        phis = np.concatenate([walkers(sp, "random")] * (nw // 2))
        got.append({call: (phi[:2], ld[:2]) for call, (phi, ld) in calls(sys_, phis, "random").items()})
        sys_.close()
    for call in got[0]:
        assert np.array_equal(got[0][call][0], got[1][call][0]), call
        assert np.array_equal(got[0][call][1], got[1][call][1]), call


def gradient_bounds(osys, phi, g1):
    """Sums of absolute values behind dE/dphi = [S^-1 (Gam - (Gam phi S^-1) A^dag)]^H of E1 and behind dE/dh, one
    walker: the scale of one relative rounding of every operand."""
    Ad, nk = osys.A_dense(), osys.nk
    bphi, bh = np.empty(phi.shape), np.zeros((nk, osys.M, osys.M))
    for s in range(2):
        Gam = np.zeros((osys.N, osys.NM))
        for k in range(nk):
            Gam[osys.rows(k), osys.cols(k)] = abs(g1) * np.abs(osys.A[k].conj().T @ osys.h[k])
        Sinv, p = np.abs(np.linalg.inv(Ad.conj().T @ phi[s])), np.abs(phi[s])
        bphi[s] = (Sinv @ (Gam + Gam @ p @ Sinv @ np.abs(Ad).T)).T
        Gh = (p @ Sinv).T
        for k in range(nk):
            bh[k] += abs(g1) * np.abs(osys.A[k]) @ Gh[osys.rows(k), osys.cols(k)]
    return bphi, bh


GRAD = {"N16": ((2, 2, 2), 2, 8), "N65": ((5, 1, 1), 13, 15), "N108": ((3, 3, 3), 4, 8), "N108wide": ((3, 3, 3), 4, 26),
        "N256": ((4, 4, 1), 16, 17)}
# u per kind of walkers: dE/dphi, dE/dh
#   near: S^-1 is near the identity, so one product of each sum outweighs the others and every running sum keeps its
#   size: sqrt(2 k) roundings of 2^-49 in the mean, k <= 702, 19 2^-49 per product sum, twice: u = 2^-44.
#   random: terms of random sign, running sums far below the sums of absolute values: the operands' own
#   rounding to 48 bits (2^-48 at most, half of it in the mean, and cond(S) 2^-53 of the inverse): u = 2^-48 for
#   dE/dphi, whose bound multiplies four such sums, 2^-47 for dE/dh.
GRAD_U = {"near": (2.0**-44, 2.0**-44), "random": (2.0**-48, 2.0**-47)}


@pytest.mark.parametrize("kind", list(GRAD_U))
@pytest.mark.parametrize("name", list(GRAD))
def test_e1_gradient(name, kind):
    """E1 alone: no part of its gradient passes through the 22-bit exchange or the fp32 Coulomb sum."""
    sp = spec(*GRAD[name])
    sys_, osys = make(sp, "mixed")
    phis = walkers(sp, kind)
    g = np.zeros((2, 3), dtype=np.complex128)
    g[:, 0] = gen.upstream(sp)[:, 0]
    gphi, gh1 = (host(t) for t in sys_.local_energy_backward(dev(phis), dev(g)))
    ref = [ok.local_energy_vjp(osys, phis[w], g[w], two_body=lambda *a: None) for w in range(2)]
    bounds = [gradient_bounds(osys, phis[w], g[w, 0]) for w in range(2)]
    uphi, uh = GRAD_U[kind]
    for w in range(2):
        assert np.linalg.norm(gphi[w] - ref[w][0]) < uphi * np.linalg.norm(bounds[w][0])
    assert np.linalg.norm(gh1 - sum(r[1] for r in ref)) < uh * np.linalg.norm(sum(b[1] for b in bounds))
    only = host(sys_.local_energy_backward(dev(phis), dev(g), want_phi=False)[1])
    assert np.array_equal(only, gh1)
    sys_.close()


def test_e1_gradient_weights():
    """The weights enter in FP64: with the trial itself as the walker S^-1 is the identity and the virtual rows of
    dE1/dphi are g conj(h A) unprojected, exact but for their one rounding to 48 bits (2^-48 of each
    part; an eighth more for the FP64 operations)."""
    sp = spec((2, 1, 1), 2, 24)
    sys_, osys = make(sp, "mixed")
    phis = np.broadcast_to(gen.trial_dense(sp), (2, 2, sp.NM, sp.N))
    g = np.zeros((2, 3), dtype=np.complex128)
    g[:, 0] = gen.upstream(sp)[:, 0]
    gphi = host(sys_.local_energy_backward(dev(phis), dev(g), want_h1=False)[0])
    for k in range(sp.nk):
        virtual, occupied = slice(k * sp.M + sp.nocc, (k + 1) * sp.M), osys.rows(k)
        want = g[:, 0, None, None, None] * (osys.A[k].conj().T @ osys.h[k]).conj().T[sp.nocc:]
        d = gphi[:, :, virtual, occupied] - want
        u = 1.125 * 2.0**-48
        assert (np.abs(d.real) <= u * np.abs(want.real)).all() and (np.abs(d.imag) <= u * np.abs(want.imag)).all()
    sys_.close()
