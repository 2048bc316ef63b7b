"""Sizes on both sides of every line at which a kernel or its layout changes, against the FP64 oracle.

The lines (N occupied orbitals per spin over all k-points):
  overlap inverse / log det   32, 64 (threads per matrix), 110 | 111 (one | two CTAs), 128, 256 (in shared
                              memory | in the global copy; kept for the adjoint | formed again)
  Cholesky-QR                 32, 64, 128, 256 (threads), 165 | 168 (rows in shared memory | in global),
                              512 (rows in registers | the blocked form)
  adjoint's Green's function  32- and 16-wide chunks of the contraction, odd M, odd nocc M
  FP64 LU                     78 | 80 (inverse beside the factor | factor alone in shared memory), 112 | 114
                              (factor in shared memory | in global)
  one-body exponential        squarings (time step 2), none (0.01)
Odd N, odd nocc M and odd M reach the scalar tails of the 16-byte epilogues.

Bars: those of the two paths elsewhere: FP64 1e-10; mixed on near-trial walkers 1e-6 normwise
for force bias and orbitals, 1e-5 Ha per cell, 1e-5 for weights, log det and dE/dphi, 1e-10 for dE/dh;
QR max(1e-6, 2e-7 cond(phi)) and orthonormal to 1e-6.
"""
import numpy as np
import pytest

import gen
from oracle import afqmc_kp as ok

torch = pytest.importorskip("torch")
from gpu_util import dev, host, make, oracle_energy, oracle_xbar, rel  # noqa: E402

pytestmark = pytest.mark.gpu


def spec(nk, nocc, M, nw=2, nchol=2, dt=0.01):
    return gen.SystemSpec(grid=(nk, 1, 1), M=M, nocc=nocc, nchol=nchol, nwalkers=nw, dt=dt, random_trial=True, seed=nk)


MIXED = {
    "N1": spec(1, 1, 2), "N31": spec(1, 31, 33), "N32": spec(4, 8, 9), "N33": spec(3, 11, 13),
    "N63": spec(7, 9, 11), "N64": spec(4, 16, 17), "N65": spec(5, 13, 15),
    "N110": spec(5, 22, 23), "N111": spec(37, 3, 4), "N128": spec(8, 16, 17), "N129": spec(43, 3, 4),
    "N160": spec(8, 20, 21), "N165": spec(15, 11, 12), "N168": spec(12, 14, 15),
    "N256": spec(16, 16, 17), "N258": spec(43, 6, 7),
    "G401": spec(1, 2, 3, nchol=401),   # the adjoint takes 16 walkers per block, not 32
    # more matrices than clusters of eight or four can take at once with profit: the global forms
    "N256-many": spec(16, 16, 17, nw=64), "N160-many": spec(8, 20, 21, nw=64),
    # more matrices than SMs: no doubling of the CTAs per matrix
    "N66-many": spec(3, 22, 23, nw=90),
}
QR_ONLY = {"N512": spec(32, 16, 17, nw=1, nchol=1), "N520": spec(40, 13, 14, nw=1, nchol=1)}
FP64 = {"N78": spec(6, 13, 15), "N80": spec(8, 10, 11), "N112": spec(16, 7, 9), "N114": spec(38, 3, 4),
        "long-step": spec(3, 2, 5, dt=2.0)}


@pytest.mark.parametrize("name", list(MIXED))
def test_mixed(name):
    sp = MIXED[name]
    sys_, osys = make(sp, "mixed")
    phis = gen.near_trial_walkers(sp)
    few = range(min(sp.nwalkers, 2))
    e, xb = host(sys_.local_energy(dev(phis))), host(sys_.force_bias(dev(phis)))
    ref_e = oracle_energy(osys, phis, few)
    assert np.abs(e[few] - ref_e).max() < 1e-5 * sp.nk
    assert rel(xb[few], np.array([oracle_xbar(osys, phis[w]) for w in few])) < 1e-6
    x, w0 = gen.fields(sp, 1), np.linspace(0.5, 1.5, sp.nwalkers)
    phi, w = dev(phis), dev(w0)
    ld = torch.empty((sp.nwalkers, 2), dtype=torch.complex128, device="cuda")
    sys_.propagate(phi, dev(x), w, logdet=ld)
    ref = [ok.propagate_walker(osys, phis[i], x[i], w0[i]) for i in few]
    assert rel(host(phi)[few], np.array([r[0] for r in ref])) < 1e-6
    assert rel(host(w)[few], np.array([r[1] for r in ref])) < 1e-5
    d = host(ld)[few] - np.array([r[2] for r in ref])
    assert np.abs(d.real).max() < 1e-5 and np.abs(np.angle(np.exp(1j * d.imag))).max() < 1e-5
    g = np.zeros((sp.nwalkers, 3), dtype=np.complex128)
    g[0] = gen.upstream(sp)[0]
    gphi, gh1 = sys_.local_energy_backward(dev(phis), dev(g))
    ref_phi, ref_h1 = ok.local_energy_vjp(osys, phis[0], g[0])
    assert rel(host(gphi)[0], ref_phi) < 1e-5
    assert rel(host(gh1), ref_h1) < 1e-10
    check_qr(sp, sys_, phis)
    assert sys_.last_error() == (0, 0)
    sys_.close()


def check_qr(sp, sys_, phis):
    rng = np.random.default_rng(4)
    mix = rng.standard_normal((sp.N, sp.N)) + 1j * rng.standard_normal((sp.N, sp.N))
    phis = phis[:2] @ (np.eye(sp.N) + 0.3 * mix / np.sqrt(sp.N))
    full = np.concatenate([phis] * ((sp.nwalkers + 1) // 2))[:sp.nwalkers]
    phi = dev(full)
    sys_.orthonormalise(phi)
    got = host(phi)[:len(phis)]
    ref = np.array([[ok.orthonormalise(p[s]) for s in range(2)] for p in phis])[:len(got)]
    cond = max(np.linalg.cond(p[s]) for p in phis for s in range(2))
    assert rel(got, ref) < max(1e-6, 2e-7 * cond), cond
    q = got.reshape(-1, sp.NM, sp.N)
    assert np.abs(np.einsum("bij,bik->bjk", q.conj(), q) - np.eye(sp.N)).max() < 1e-6


@pytest.mark.parametrize("name", list(QR_ONLY))
def test_qr(name):
    sp = QR_ONLY[name]
    sys_, _ = make(sp, "mixed")
    check_qr(sp, sys_, gen.near_trial_walkers(sp))
    sys_.close()


@pytest.mark.parametrize("name", list(FP64))
def test_fp64(name):
    sp = FP64[name]
    sys_, osys = make(sp, "fp64")
    phis = gen.near_trial_walkers(sp)
    assert rel(host(sys_.local_energy(dev(phis))), oracle_energy(osys, phis)) < 1e-10
    x, w0 = gen.fields(sp, 1), np.ones(sp.nwalkers)
    phi, w = dev(phis), dev(w0)
    ld = torch.empty((sp.nwalkers, 2), dtype=torch.complex128, device="cuda")
    sys_.propagate(phi, dev(x), w, logdet=ld)
    ref = [ok.propagate_walker(osys, phis[i], x[i], w0[i]) for i in range(sp.nwalkers)]
    assert rel(host(phi), np.array([r[0] for r in ref])) < 1e-10
    d = host(ld) - np.array([r[2] for r in ref])
    assert np.abs(d.real).max() < 1e-10 * max(1.0, np.abs(host(ld)).max())
    sys_.close()
