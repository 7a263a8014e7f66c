"""Edges of the kernels' own forms: the FP16 pairs of scaled fields (tensor-core
Step II), the moment counts of the binning's warp sums, views binned together, and
the shell fields packed two to a transform."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2405_14513_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_14513_gb300 import api  # noqa: E402


def _floored(got, ref):
    fin = np.isfinite(ref)
    assert np.array_equal(fin, np.isfinite(got))
    g, r = (np.where(fin, x, 0.0).reshape(-1, ref.shape[-1]) for x in (got, ref))
    floor = np.maximum(1e-2 * np.abs(r).max(axis=0, keepdims=True), 1e-300)
    return (np.abs(g - r) / np.maximum(np.abs(r), floor)).max()


@pytest.mark.parametrize("ng,k", [(12, -24), (32, 20), (48, -40), (64, 30)])
def test_power_of_two_amplitudes_are_exact(ng, k):
    """Every step is exact under a factor 2^k (the stored fields are brought to one
    range, the FP16 pairs split there): B(2^k delta) = 2^(3k) B(delta), bit for bit."""
    L = 10.0 * ng
    edges = synth.default_k1_edges(ng, L, 3)
    plan = api.Plan(ng, L, edges, 4, 4, 6, precision="mixed_tc")
    ws = plan.workspace()
    d = torch.from_numpy(synth.make_field(ng, L, 3).astype(np.float32)).cuda()
    a = plan.estimate(d, ws).cpu().numpy()
    b = plan.estimate(d * 2.0 ** k, ws).cpu().numpy()
    assert plan.workspace_status(ws) == 0
    assert np.array_equal(a * 2.0 ** (3 * k), b, equal_nan=True)


@pytest.mark.parametrize("ng", [32, 96, 192])
def test_point_field_reaches_the_fp16_bound(ng):
    """A point field: every mode of a ring in phase at one grid point, where the
    stored fields, and their products, take the largest values the scaling allows.
    B_0^0 = a^3 / V in every bin; 1e-5: FP32 transforms and 2^-24 pairs, summed
    without cancellation."""
    L = 10.0 * ng
    d = np.full((ng,) * 3, -1.0 / ng ** 3)
    d[3, ng // 2, ng - 1] += 1.0
    plan = api.Plan(ng, L, synth.default_k1_edges(ng, L, 4), 4, 4, 2, precision="mixed_tc")
    B = plan.estimate(torch.from_numpy(d.astype(np.float32)).cuda(), plan.workspace()).cpu().numpy()[0]
    a = (L / ng) ** 3                            # Delta of a unit point is V / N^3 times a phase
    want = a ** 3 / L ** 3
    b00 = B[..., 0][np.isfinite(B[..., 0])]
    assert b00.size and np.abs(b00 / want - 1.0).max() < 1e-5


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4), ("mixed_tc", 1e-4), ("fp32", 1e-4)])
@pytest.mark.parametrize("l_max", [0, 2, 4, 8])
def test_moment_counts(precision, tol, l_max):
    """1, 4, 9 and 25 moments (16 are tested elsewhere): the binning's exchange of
    sums across a warp, padded to a power of two, on bins from one record to many."""
    ng, L = 16, 200.0
    edges = synth.default_k1_edges(ng, L, 2)
    field = synth.make_field(ng, L, 5).astype(np.float64 if precision == "fp64" else np.float32)
    ref = O.select_even(O.estimate(field.astype(np.float64), L, edges, 3, 2, l_max)["B"], l_max)
    plan = api.Plan(ng, L, edges, 3, 2, l_max, precision=precision)
    B = plan.estimate(torch.from_numpy(field).cuda(), plan.workspace()).cpu().numpy()[0]
    assert _floored(B, ref) < tol


@pytest.mark.parametrize("ng,l_max", [(16, 0), (24, 4), (32, 2)])
def test_shell_fields_in_pairs(ng, l_max):
    """(shells - 1) (l_max/2 + 1) real fields, an odd number among them, share
    complex transforms: B_l^0 against the oracle."""
    L = 10.0 * ng
    edges = synth.default_k1_edges(ng, L, 2)
    field = synth.make_field(ng, L, 9).astype(np.float32)
    ref = O.shell_estimate(field.astype(np.float64), L, edges, 3, 3, l_max)
    plan = api.ShellPlan(ng, L, edges, 3, 3, l_max)
    B = plan.estimate(torch.from_numpy(field).cuda(), plan.workspace()).cpu().numpy()
    assert _floored(B, ref) < 1e-4


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed_tc"])
@pytest.mark.parametrize("ng,bins", [(12, [3, 1]), (24, [2, 2, 1]), (32, [9, 5, 3, 2, 1]), (32, [2, 3, 3, 4, 4])])
def test_views_binned_together(precision, ng, bins):
    """Views of every l_hi, of few and of many bins, binned in one launch, two fields
    at once: each equals, bit for bit, the same moments of a plan with that one view."""
    L, l_max = 10.0 * ng, 2 * len(bins) - 2
    edges = synth.default_k1_edges(ng, L, 3)
    dt = np.float64 if precision == "fp64" else np.float32
    d = torch.from_numpy(np.stack([synth.make_field(ng, L, s).astype(dt) for s in (7, 8)])).cuda()
    plan = api.Plan(ng, L, edges, 1, 1, l_max, precision=precision, mu_t_bins_l=bins, max_batch=2)
    assert len(plan.views) == len(set(bins))
    ws = plan.workspace(2)
    blocks = plan.split(plan.estimate(d, ws).cpu().numpy())
    assert plan.workspace_status(ws, 2) == 0
    for v, blk in zip(plan.views, blocks):
        one = api.Plan(ng, L, edges, v["n_mu"], v["n_t"], l_max, precision=precision, max_batch=2)
        want = one.estimate(d, one.workspace(2)).cpu().numpy()
        lo = (v["l_lo"] // 2) ** 2
        assert np.array_equal(blk, want[..., lo:lo + v["n_lm"]], equal_nan=True), v
        one.close()
    plan.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_tc"])
@pytest.mark.parametrize("ng", [8, 32, 64])
def test_back_to_back_estimates_wait_for_each_other(precision, ng):
    """The kernels of an estimate are placed before the ones ahead of them end: forty
    estimates of alternating fields in one workspace, the input written by the kernel
    ahead and the output read by the one behind, none synchronised, give the bits of
    single ones."""
    L = 10.0 * ng
    dt = torch.float64 if precision == "fp64" else torch.float32
    plan = api.Plan(ng, L, synth.default_k1_edges(ng, L, 2), 4, 4, 4, precision=precision)
    ws = plan.workspace()
    fields = [torch.from_numpy(synth.make_field(ng, L, s)).to("cuda", dt) for s in (1, 2)]
    want = []
    for f in fields:
        want.append(plan.estimate(f, ws).cpu().numpy())
    buf = torch.empty_like(fields[0])
    got = []
    for i in range(40):
        buf.copy_(fields[i % 2])
        got.append(plan.estimate(buf, ws).clone())
        buf.zero_()
    for i, g in enumerate(got):
        assert np.array_equal(g.cpu().numpy(), want[i % 2], equal_nan=True), i
    plan.close()
