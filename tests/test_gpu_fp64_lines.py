"""FP64 path on both sides of the lines at which lu_kernel's layout changes, against the oracle at 1e-10.

The factor and, for the inverse, the solution lie in shared memory while they take 200 KiB at most: 2 x 16 N^2
up to N = 80, 16 N^2 up to N = 113 (112 and 114 are the nearest sizes that a handle takes).  The energy needs the
inverse, the log det of the propagated walkers the factor alone; the weight sums the force bias.
"""
import numpy as np
import pytest

import gen
from oracle import afqmc_kp as ok

torch = pytest.importorskip("torch")
from gpu_util import dev, host, make, oracle_energy, rel, wrap_phase  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = {"N1": ((1, 1, 1), 1, 2), "N80": ((4, 4, 1), 5, 6), "N81": ((3, 3, 3), 3, 4), "N112": ((4, 2, 2), 7, 8),
         "N114": ((19, 2, 1), 3, 4)}


@pytest.mark.parametrize("name", list(SIZES))
def test_fp64_lines(name):
    grid, nocc, M = SIZES[name]
    sp = gen.SystemSpec(grid=grid, M=M, nocc=nocc, nchol=3, nwalkers=2, dt=0.01, random_trial=True, seed=7)
    sys_, osys = make(sp, "fp64")
    phis = gen.near_trial_walkers(sp)
    assert rel(host(sys_.local_energy(dev(phis))), oracle_energy(osys, phis)) < 1e-10
    x, w0 = gen.fields(sp, 2), np.array([0.75, 1.5])
    phi, w = dev(phis), dev(w0)
    ld = torch.empty((2, 2), dtype=torch.complex128, device="cuda")
    sys_.propagate(phi, dev(x), w, logdet=ld)
    ref = [ok.propagate_walker(osys, phis[i], x[i], w0[i]) for i in range(2)]
    assert rel(host(phi), np.array([r[0] for r in ref])) < 1e-10
    assert rel(host(w), np.array([r[1] for r in ref])) < 1e-10
    d = host(ld) - np.array([r[2] for r in ref])
    assert max(np.abs(d.real).max(), np.abs(wrap_phase(d.imag)).max()) < 1e-10
    assert sys_.last_error() == (0, 0)
    sys_.close()
