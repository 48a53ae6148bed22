"""The cluster shapes of the GPU discrete velocity method against the oracle: columns that do not
divide by the CTAs or the warps, one to many nodes a lane, one instance to more than the card has SMs
for, and state buffers that only fit when split."""
import numpy as np
import pytest

import oracle
from lbtest import lib

pytestmark = pytest.mark.gpu

U0 = 1e-3


@pytest.mark.parametrize("n,nx,count,nsteps", [(2, 3, 1, 60), (3, 9, 2, 60), (20, 33, 1, 70), (64, 40, 1, 40),
                                               (5, 130, 20, 65), (8, 64, 200, 33), (64, 440, 100, 5), (2, 7200, 1, 3)])
def test_every_cluster_shape_matches_oracle(n, nx, count, nsteps):
    """1e-12 of the amplitude a level, the bound of the other comparisons of the two FP64 codes."""
    Lattice, capi = lib()
    taus = np.geomspace(0.02, 2.0, count)
    amp, phi = 1e-3, 0.7
    A, S = capi.lb_dvm_run_forced(taus, n, nx, U0, amp, phi, nsteps)
    for i in sorted({0, count // 2, count - 1}):
        _, Ao, So = oracle.run_dvm(n, nx, taus[i], U0, nsteps, kn_convention="paper", force_amp=amp, force_freq=phi)
        scale = max(np.max(np.abs(Ao)), amp)
        assert np.max(np.abs(A[i] - Ao)) < 1e-12 * scale * (nsteps + 1)
        assert np.max(np.abs(S[i] - So)) < 1e-12 * scale * (nsteps + 1)
