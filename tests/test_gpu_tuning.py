"""What the creation of a context costs beyond its own fields: timings are taken once per process and
lattice shape."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1410_7170_gb300 as ovl  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_7170_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def test_second_context_of_a_shape_launches_no_timings():
    dims = (8, 4, 4, 12)
    U = synth.gauge_field(dims, 0.5, 61)

    def create(**kw):
        op = ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(
            lambda_min=0.2, lambda_max=8.0, m0_prec=-0.25, precision=ovl.OVL_MIXED_FP32, precond=ovl.OVL_PREC_WILSON,
            sap_block=(2, 2, 2, 2), **kw))
        n, ms = op.prof_get()["launches"], op.tuning_sap()["ms"]
        op.close()
        return n, ms

    first, ms = create()
    again, ms2 = create()
    bare, _ = create(stencil_tps=1, mrhs_kernel=1, sap_tps=1)   # every choice made by the caller
    assert again == bare < first
    assert min(ms) > 0 and ms2 == ms
