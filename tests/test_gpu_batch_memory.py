"""hbs_build_batch when the device runs out of memory while periodizers and compression run beside one another:
the batch is built once more, one periodizer after another."""
import numpy as np
import pytest

from gpu_util import relerr, require_lib
from paper_1301_1247_gb300 import inputs

pytestmark = pytest.mark.gpu

THETA = [-0.7, -2.0]


def _batch(hbs):
    geoms = [inputs.star(0.25, 0.2, 5).sample(n) for n in (400, 900, 1500)]
    return hbs.build_batch(geoms, [10.0, 12.0, 20.0], 1.0, 1e-12)


def _amplitudes(handles):
    return np.concatenate([np.concatenate(r.bragg(i)[1:3]) for r in (h.solve(THETA) for h in handles) for i in range(r.n)])


@pytest.mark.parametrize("after", [0, 40, 200, 400])
def test_a_full_device_is_met_by_a_second_attempt(after):
    """The failure in the geometry, in the compression or in a periodizer: the solvers are those of a normal
    build (1e-11, the bound of the library's comparison of batch and single builds)."""
    hbs = require_lib()
    want = _amplitudes(_batch(hbs))
    hbs.fault_inject(hbs.INJECT_DEVICE_FULL, after)
    try:
        got = _amplitudes(_batch(hbs))
    finally:
        hbs.fault_inject(hbs.INJECT_CLEAR)
    assert relerr(got, want) < 1e-11


@pytest.mark.parametrize("kind", ["INJECT_ALLOC_FAILURE", "INJECT_DEVICE_FULL"])
def test_failures_that_are_reported(kind):
    """An allocation failure of a batch, and a full device under a single build, give HBS_ERR_OOM; the next build
    works."""
    hbs = require_lib()
    hbs.fault_inject(getattr(hbs, kind), 60)
    try:
        with pytest.raises(hbs.HbsError) as e:
            if kind == "INJECT_ALLOC_FAILURE":
                _batch(hbs)
            else:
                hbs.Handle(*inputs.star(0.25, 0.2, 5).sample(400), 1.0, 10.0, 1e-12)
        assert e.value.status == hbs.HBS_ERR_OOM
    finally:
        hbs.fault_inject(hbs.INJECT_CLEAR)
    assert np.all(np.isfinite(_amplitudes(_batch(hbs))))
