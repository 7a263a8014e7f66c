"""The FP32 forward transform's amplitudes: no systematic loss beyond half a unit in the
last place, which every triple product would take three times."""
import numpy as np
import pytest

from paper_2405_14513_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_14513_gb300 import api  # noqa: E402


@pytest.mark.parametrize("ng", [24, 48, 64, 96])
def test_amplitudes(ng):
    """Mean over the modes within the rings of Re(error / Delta), weighted by |Delta|^2,
    over four fields, against FP64: at most 2^-24."""
    L = 10.0 * ng
    plan = api.Plan(ng, L, synth.default_k1_edges(ng, L, 2), 2, 2, 0, precision="fp32")
    ws = plan.workspace()
    nz = ng // 3
    f = np.rint(np.fft.fftfreq(ng) * ng)
    inside = 9 * (f[:, None] ** 2 + f[None, :] ** 2) < ng * ng
    num = den = 0.0
    for seed in range(4):
        d = synth.make_field(ng, L, 40 + seed).astype(np.float32)
        plan.estimate(torch.from_numpy(d).cuda(), ws)
        ref = np.fft.fftn(d.astype(np.float64)) * (L / ng) ** 3
        ref[0, 0, 0] = 0.0
        for n in range(nz + 1):
            x, e = ref[:, :, n][inside], (plan.delta_plane(ws, n) - ref[:, :, n])[inside]
            num += float(np.sum(e * x.conj()).real)
            den += float(np.sum(np.abs(x) ** 2))
    assert abs(num / den) < 2.0 ** -24
