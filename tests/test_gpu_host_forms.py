"""The two host-memory forms of an estimate on one plan, in either order: each makes the
buffers that it finds missing."""
import numpy as np
import pytest

from paper_2405_14513_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_14513_gb300 import api  # noqa: E402


@pytest.mark.parametrize("first", ["submit", "call"])
def test_host_forms_in_either_order(first):
    ng, L = 16, 160.0
    plan = api.Plan(ng, L, synth.default_k1_edges(ng, L, 2), 3, 3, 2, precision="mixed")
    d = synth.make_field(ng, L, 2).astype(np.float32)[None]
    want = plan.estimate(torch.from_numpy(d).cuda(), plan.workspace()).cpu().numpy()
    plan.close()
    plan = api.Plan(ng, L, synth.default_k1_edges(ng, L, 2), 3, 3, 2, precision="mixed")
    stream = torch.cuda.current_stream()

    def submit():
        out = np.empty(plan.out_doubles)
        plan.host_submit(d, out, stream=stream)
        return plan.host_wait().reshape(want.shape)

    forms = [submit, lambda: plan.estimate_host(d)]
    for f in forms if first == "submit" else forms[::-1]:
        assert np.array_equal(f(), want, equal_nan=True)
    plan.close()


def test_a_failed_allocation_is_not_the_next_calls_error():
    """A workspace of terabytes is refused; the estimate after it is not."""
    ng, L = 64, 640.0
    plan = api.Plan(ng, L, synth.default_k1_edges(ng, L, 2), 2, 2, 0, precision="mixed", max_batch=65535)
    assert plan.workspace_bytes(65535) > 1 << 40
    d = synth.make_field(ng, L, 2).astype(np.float32)[None]
    with pytest.raises(api.BispError) as e:
        plan.estimate_host(d)
    assert e.value.status == 3                       # BISP_OUT_OF_MEMORY
    B = plan.estimate(torch.from_numpy(d).cuda(), plan.workspace(1)).cpu().numpy()
    assert np.isfinite(B).any()
    plan.close()
