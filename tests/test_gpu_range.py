"""The tensor-core Step II on fields whose values differ by orders of magnitude within a
ring: the FP16 pairs hold small values to 2^-25 of the scale that the largest set."""
import numpy as np
import pytest

from paper_2405_14513_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_14513_gb300 import api  # noqa: E402


def _field(kind, ng, L):
    d = synth.make_field(ng, L, 5)
    rng = np.random.default_rng(8)
    if kind == "point":                   # one point on a field a millionth of it
        d = 1e-6 * d
        d[3, ng // 2, ng - 1] += 1.0
    elif kind == "lognormal":             # a few points hold most of the field
        y = np.exp(3.0 * rng.standard_normal((ng,) * 3))
        d = y / y.mean() - 1.0
    elif kind == "slab":                  # an eighth of the box 10^4 times the rest
        d = d * np.where(np.arange(ng) < ng // 8, 1.0, 1e-4)[:, None, None]
    return (d - d.mean()).astype(np.float32)


@pytest.mark.parametrize("kind", ["point", "lognormal", "slab"])
@pytest.mark.parametrize("ng", [24, 64])
def test_values_of_all_sizes(kind, ng):
    """Triple sums of mixed_tc against FP64, 2-norm over the combinations: three FP32
    fields of a relative error of 1e-6 at most, so 3e-6."""
    L = 10.0 * ng
    edges = synth.default_k1_edges(ng, L, 3)
    d = torch.from_numpy(_field(kind, ng, L)).cuda()
    S = []
    for precision in ("mixed_tc", "fp64"):
        plan = api.Plan(ng, L, edges, 4, 4, 2, precision=precision)
        ws = plan.workspace()
        plan.estimate(d.double() if precision == "fp64" else d, ws)
        ints = plan.combo_table()["ints"]
        order = np.lexsort(ints.T)
        S.append((ints[order], plan.combo_sums(ws)[order]))
    assert np.array_equal(S[0][0], S[1][0])
    assert np.linalg.norm(S[0][1] - S[1][1]) < 3e-6 * np.linalg.norm(S[1][1])
