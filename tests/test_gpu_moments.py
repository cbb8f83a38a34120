"""Moments of all power combinations of a shell pair at once, against the oracle: orders around the passes of the
kernel (256 sums each), the doubled panels above n = 32, shells of one kind and mixed, a box that misses some pairs.
Tolerance: 1e-13 of the plan's largest moment of each dimension, as for screened plans in test_gpu_parity.py (a
product centred outside the box has moments far below that, cut where its Gaussian falls below exp(-81))."""
import numpy as np
import pytest

import oracle
from paper_2210_13069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shells", [(("s", 2),), (("p", 1),), (("s", 1), ("p", 1), ("d", 1))])
@pytest.mark.parametrize("n", [1, 2, 28, 29, 32, 33, 64])
def test_moment_groups(n, shells):
    from paper_2210_13069_gb300 import build_lib, lrtei
    build_lib.build()
    lrtei.load()
    m = synth.random_molecule(77, natoms=2, cube=3.0, shells_per_atom=shells, nprim=2, alpha_range=(0.1, 200.0),
                              omega=0.5, n=n, P=3)
    c = m.atoms[0]
    m.box_lo, m.box_hi = c - 1.5, c + 1.5
    o = oracle.Oracle.from_molecule(m)
    pl = lrtei.Plan(m, "fp64")
    S = pl.factors()[0].cpu().numpy()
    top = np.abs(S).max(axis=(1, 2))
    row = 0
    for mu in range(m.nbf):
        for nu in range(mu, m.nbf):
            W = [o.moments(mu, nu, d) for d in range(3)]
            for d in range(3):
                assert np.all(np.abs(S[d, row:row + W[d].shape[0]] - W[d]) <= 1e-13 * top[d]), (mu, nu, d)
            row += W[0].shape[0]
    assert row == S.shape[1]
    pl.close()
