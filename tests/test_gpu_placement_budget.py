"""A budget of exactly one solve's footprint admits placement, voxelization and that solve: the fixed
scratch of a context (64 KB, sphere lists and filter buffers) stays outside the budget."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg, inputs as I


def test_placement_beside_a_full_budget():
    N, n, f = 8, 100, 0.40
    ref = I.generate_spheres(3000, n, f).spheres
    with hmg.Context(0, hmg.hmg_footprint(N, hmg.HMG_FP64)) as c:
        for _ in range(2):   # before the solve state exists and beside it
            got, _ = hmg.hmg_rsa(c.handle, 3000, n, I.sphere_radius(n, f))
            assert np.array_equal(got, ref)
            ph = np.empty(N ** 3, dtype=np.uint8)
            hmg.hmg_voxelize(c.handle, ref, 0.3, N, ph)
            K, _, _ = hmg.hmg_solve(c.handle, ph, N, (0.2, 0.25, 2.0), 1e-6, hmg.HMG_FP64)
            assert np.isfinite(K).all()
    with hmg.Context(0, 1000) as c:   # the centres themselves are counted
        with pytest.raises(hmg.HmgError) as ex:
            hmg.hmg_rsa(c.handle, 3000, n, I.sphere_radius(n, f))
        assert ex.value.status == hmg.HMG_OUT_OF_MEMORY
