"""The allocation-free entry point at the sizes where its launches change (the lane
rule's limits, grids with a part-filled last block, the capacity) and for every
species count, against the ordinary path; the tolerance is that of its other tests.
Collected after the others, as the tests of the entry point are."""

import numpy as np
import pytest

import workloads as W
from gpu_common import TOL_FORCE, normwise
from test_zz_no_alloc import _noalloc_forces, _reference_forces

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('n, ns, L, s_f', [
    (1, 1, 5.0, 2.0), (33, 4, 5.0, 2.0), (1500, 2, 7.3, 2.0), (1501, 3, 7.3, 1.0), (6000, 4, 11.4, 2.0),
    (6001, 1, 11.4, 1.0), (16384, 2, 12.5, 2.0)])
def test_sizes_and_species(n, ns, L, s_f):
    d = W.fluid_box(L=L, rho=1.1 * n / L ** 3 + 1.0, n_species=ns, seed=900 + n % 97, s_f=s_f)
    d['kappa'][...] = np.linspace(0.4, 1.6, ns, dtype=np.float32)
    p = d['particles']
    assert p['pos'].shape[0] >= n
    d['particles'] = {k: np.ascontiguousarray(v[:n]) for k, v in p.items()}
    F, Q = _noalloc_forces(d)
    Fr, Qr = _reference_forces(d)
    assert np.isfinite(F).all() and np.isfinite(Q).all()
    if n == 1:
        assert not F.any() and not Q.any() and not Fr.any()
    else:
        assert normwise(F, Fr) < TOL_FORCE
        assert normwise(Q, Qr) < TOL_FORCE
