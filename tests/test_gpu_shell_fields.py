"""The shell estimator's fields and triple sums one by one, against 64 bits from the
same planes of Delta (the first array of the workspace): each real field has the
rounding error of its own size, whatever the fields beside it hold."""
import numpy as np
import pytest

from paper_2405_14513_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_14513_gb300 import api  # noqa: E402


def _shells(ng):
    """Shell of every mode, and the modes (FFT order)."""
    e3 = [0]
    while e3[-1] < ng:
        e3.append(min(e3[-1] + (3 << ((len(e3) - 1) // 10)), ng))
    f = torch.fft.fftfreq(ng, d=1.0 / ng, dtype=torch.float64, device="cuda").round().long()
    q = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
    shell = torch.bucketize(9 * q, torch.tensor([e * e for e in e3], device="cuda"), right=True) - 1
    return shell, f, q, len(e3) - 1


def _reference(plan, ws):
    """num[t][l], and the 2-norm of the products it adds, from the workspace's Delta."""
    ng, nz = plan.n_g, plan.n_g // 3
    planes = ws[:(nz + 1) * ng * ng * 8].view(torch.float32).double().reshape(nz + 1, ng, ng, 2)
    half = torch.view_as_complex(planes.contiguous()).permute(1, 2, 0)                     # [a][b][n]
    D = torch.zeros((ng,) * 3, dtype=torch.complex128, device="cuda")
    D[:, :, :nz + 1] = half
    D[:, :, ng - nz:] = torch.roll(torch.flip(half[:, :, 1:], (0, 1, 2)), (1, 1), (0, 1)).conj()
    shell, f, q, ns = _shells(ng)
    mu = f[None, None, :] / torch.sqrt(q.clamp(min=1).double())
    P = [torch.ones_like(mu), (3 * mu ** 2 - 1) / 2, (35 * mu ** 4 - 30 * mu ** 2 + 3) / 8,
         (231 * mu ** 6 - 315 * mu ** 4 + 105 * mu ** 2 - 5) / 16][:plan.nl]
    Y = [((4 * i + 1) / (4 * np.pi)) ** 0.5 * p for i, p in enumerate(P)]
    G = [torch.fft.fftn(torch.where(shell == s, D, 0.0)).real.reshape(-1) for s in range(ns)]
    F = [[torch.fft.fftn(torch.where(shell == s, D * y, 0.0)).real.reshape(-1) for y in Y] for s in range(ns)]
    num, norm = np.zeros((plan.n_triples, plan.nl)), np.zeros((plan.n_triples, plan.nl))
    for t, (a, b, c, _) in enumerate(plan.triples()["tri"]):
        gg = G[b] * G[c]
        for i in range(plan.nl):
            p = F[a][i] * gg
            num[t, i], norm[t, i] = float(p.sum()) / ng ** 3, float(p.norm()) / ng ** 3
    return num, norm


@pytest.mark.parametrize("ng,l_max", [(12, 0), (24, 4), (32, 0), (48, 4), (64, 6), (128, 0)])
def test_shell_fields_keep_their_own_error(ng, l_max):
    """Every third shell a thousand times its neighbours.  A field's transform has a
    relative error of at most 1e-6 (2-norm), so the error of a triple's sum, over the
    2-norm of its products, is about sqrt(3) of that at most: 2e-6 rms over the triples.
    A shell that took its neighbour's error would show 1e-4."""
    L = 10.0 * ng
    shell, _, _, _ = _shells(ng)
    w = torch.fft.fftn(torch.from_numpy(synth.make_field(ng, L, 3)).cuda().double())
    d = torch.fft.ifftn(torch.where(shell % 3 == 1, 1000.0 * w, w)).real.float().contiguous()
    plan = api.ShellPlan(ng, L, synth.default_k1_edges(ng, L, 3), 3, 3, l_max)
    ws = plan.workspace()
    plan.estimate(d, ws)
    num = plan.sums(ws)
    ref, norm = _reference(plan, ws)
    err = np.sqrt(np.mean(((num - ref) / norm) ** 2, axis=0))
    assert err.max() < 2e-6, err


@pytest.mark.parametrize("ng", [24, 32, 64])
def test_shell_sums_reach_the_largest_products(ng):
    """Three plane waves, k1 + k2 + k3 = 0, in shells 7, 5 and 4: D = V a cos(k x) in
    each, so num_l = Y_l0(0) (V a)^3 / 4, with products up to 0.9 of FP32's largest: no
    product overflows, and their sums are FP64's.  1e-5: three FP32 fields of 1e-6."""
    L = 1e4
    a = (0.9 * 3.4028234e38) ** (1 / 3) / L ** 3
    x = np.arange(ng) * (2 * np.pi / ng)
    d = sum(a * np.cos(i * x[:, None] + j * x[None, :]) for i, j in ((7, 0), (-4, 3), (-3, -3)))
    d = torch.from_numpy(np.repeat(d[:, :, None], ng, axis=2).astype(np.float32)).cuda()
    plan = api.ShellPlan(ng, L, np.array([3.0, ng / 3.0]) * (2 * np.pi / L), 1, 1, 6)
    ws = plan.workspace()
    plan.estimate(d, ws)
    num = plan.sums(ws)
    t = [k for k, q in enumerate(plan.triples()["tri"]) if tuple(q[:3]) == (7, 5, 4)]
    assert len(t) == 1
    y = np.sqrt((4 * np.arange(4) + 1) / (4 * np.pi)) * np.array([1.0, -1 / 2, 3 / 8, -5 / 16])
    want = y * (L ** 3 * a) ** 3 / 4
    assert np.isfinite(num[t[0]]).all()
    assert np.abs(num[t[0]] / want - 1).max() < 1e-5
