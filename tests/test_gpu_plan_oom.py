"""A tuning change whose larger buffers cannot be allocated: the call reports
it, no pass runs on the plan without its buffers, and the descriptor pass makes
the context usable again."""
import numpy as np
import pytest

from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("before", [0, 1])
def test_failed_replan_needs_the_descriptors_again(scgr_lib, before):
    X = np.ascontiguousarray(synth.mild(n=20000).X, np.float32)
    with Gpu(X, X, p=2.0, E=10) as g:
        want = g.forces()
        scgr.scgr_run(g.ctx, before)
        try:
            scgr.scgr_debug_fail_allocations(1)
            with pytest.raises(scgr.ScgrError) as e:
                scgr.scgr_set_tuning(g.ctx, scgr.SCGR_TUNE_FORCE_SPLITS, 4096)  # a split a tile: larger partials
            assert e.value.status == 4  # SCGR_ERR_OOM
        finally:
            scgr.scgr_debug_fail_allocations(0)
        for call in (lambda: scgr.scgr_run(g.ctx, 2), g.forces, lambda: scgr.scgr_step_partials(g.ctx)):
            with pytest.raises(scgr.ScgrError) as e:
                call()
            assert "descriptors" in str(e.value)
        scgr.scgr_compute_descriptors(g.ctx)
        np.testing.assert_allclose(g.forces(), want, rtol=1e-3, atol=1e-3 * np.abs(want).max())
        scgr.scgr_run(g.ctx, 2)
        assert scgr.scgr_get_result(g.ctx).iterations == 2
