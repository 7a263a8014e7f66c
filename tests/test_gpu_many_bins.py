"""The binning's last pass where bins are more than its blocks: empty bins, bins of a
chunk or two and a bin of many chunks in one block, against 64 bits and against plans of
few bins, bit for bit."""
import numpy as np
import pytest

from paper_2405_14513_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_14513_gb300 import api  # noqa: E402

FIN_BLOCKS = 16384                     # kFinBlocks of csrc/plan.hpp


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed_tc"])
@pytest.mark.parametrize("extra", [0, 1, 3 * FIN_BLOCKS])
def test_one_full_bin_among_empty_ones(precision, extra):
    """All combinations in the last of FIN_BLOCKS + extra bins (the others lie below
    every k1), two fields: the bits of a plan with that bin alone."""
    ng, L, lmax = 32, 320.0, 4
    kf = 2 * np.pi / L
    dt = torch.float64 if precision == "fp64" else torch.float32
    d = torch.from_numpy(np.stack([synth.make_field(ng, L, s) for s in (1, 2)])).to("cuda", dt)
    edges = np.append(np.linspace(0.0, 0.5 * kf, FIN_BLOCKS + extra), ng / 3 * kf)
    many = api.Plan(ng, L, edges, 1, 1, lmax, precision=precision, max_batch=2)
    one = api.Plan(ng, L, edges[-2:], 1, 1, lmax, precision=precision, max_batch=2)
    assert many.n_bins == FIN_BLOCKS + extra and many.n_combos == one.n_combos > 64 * 8
    B = many.estimate(d, many.workspace(2)).cpu().numpy()
    W = one.estimate(d, one.workspace(2)).cpu().numpy()
    assert np.isnan(B[:, :-1]).all()
    assert np.isfinite(W).all() and np.array_equal(B[:, -1], W[:, 0])
    assert np.array_equal(many.denominator()[-1], one.denominator()[0])


@pytest.mark.parametrize("l_max", [0, 2, 8])
def test_bins_of_few_combinations(l_max):
    """FP64, 160 x 160 bins: the estimates against the sums of their combinations."""
    ng, L, n = 24, 240.0, 160
    kf = 2 * np.pi / L
    plan = api.Plan(ng, L, np.array([1.0, ng / 3]) * kf, n, n, l_max, precision="fp64")
    assert plan.n_bins > FIN_BLOCKS
    ws = plan.workspace()
    B = plan.estimate(torch.from_numpy(synth.make_field(ng, L, 6)).cuda().double(), ws).cpu().numpy().reshape(-1, plan.n_lm)
    S, tab = plan.combo_sums(ws), plan.combo_table()
    mult = np.where((tab["ints"][:, 0] == 0) & (tab["ints"][:, 1] == 0), 1.0, 2.0)
    num = np.bincount(tab["bin"], weights=mult * S, minlength=plan.n_bins)        # l = 0: Y = 1 / sqrt(4 pi)
    nt = np.bincount(tab["bin"], weights=mult * tab["ntri"], minlength=plan.n_bins)
    with np.errstate(invalid="ignore", divide="ignore"):
        want = np.where(nt > 0, num / (L ** 3 * ng ** 2 * nt), np.nan)
    assert np.array_equal(np.isfinite(want), np.isfinite(B[:, 0]))
    assert (nt > 0).sum() > 500 and (nt == 0).sum() > FIN_BLOCKS
    f = nt > 0
    # FP64 sums of at most a few hundred terms, relative to the terms' sizes
    size = np.bincount(tab["bin"], weights=mult * np.abs(S), minlength=plan.n_bins)[f] / (L ** 3 * ng ** 2 * nt[f])
    assert (np.abs(B[f, 0] - want[f]) <= 1e-12 * size).all()


def test_resident_bytes_of_a_bin():
    """On the device a bin is its first chunk (8 bytes) and its moments' denominators."""
    ng, L, lmax, n = 16, 160.0, 2, 50000
    kf = 2 * np.pi / L
    edges = np.append(np.linspace(0.0, 0.5 * kf, n), ng / 3 * kf)
    many, one = (api.Plan(ng, L, e, 1, 1, lmax, precision="mixed") for e in (edges, edges[-2:]))
    assert many.n_bins == n and many.n_combos == one.n_combos
    assert many.info["resident_bytes"] - one.info["resident_bytes"] <= (n - 1) * (8 + 8 * many.n_lm) + 64
