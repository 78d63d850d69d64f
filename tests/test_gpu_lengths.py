"""GPU: the transforms at the compiled lengths that the other tests' grids do
not reach: the shell passes on sum grids of 192, 384 and 512 (and the
export of their modes at 128 and 384), and the per-object
x-pass at 128, 256, 384 and 512."""
import math

import numpy as np
import pytest

import mockgen
from tests.helpers import P_TOL, p_errors, to_device
from tests.test_gpu_bispectrum import B_TOL, SN_TOL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _monopole(F, Fw, bs, assign, b):
    """The triangles, N_T, T_0 and N_0 of the gridded fields, by torch's FP64 transforms."""
    N, S = F.shape[0], bs[3]
    n = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device="cuda")
    nx = n[:N // 2 + 1].abs()
    win = [torch.sinc(v / N) ** assign for v in (n[:, None, None], n[None, :, None], nx[None, None, :])]
    n2 = n[:, None, None] ** 2 + n[None, :, None] ** 2 + nx[None, None, :] ** 2
    F0, Fw0 = (torch.fft.rfftn(f) / win[0] / win[1] / win[2] for f in (F, Fw))
    wt = torch.where(nx > 0, 2.0, 1.0)[None, None, :]
    fields, ones, mean = [], [], []
    for s in range(S):
        c = bs[0] + s * bs[1]
        sel = (n2 >= (c - 0.5 * bs[2]) ** 2) & (n2 < (c + 0.5 * bs[2]) ** 2)
        fields.append(torch.fft.irfftn(torch.where(sel, F0, 0), (N,) * 3) * float(N) ** 3)
        ones.append(torch.fft.irfftn(sel.to(F0.dtype), (N,) * 3) * float(N) ** 3)
        w = (wt * sel).sum()
        mean.append(float((wt * sel * (F0 * Fw0.conj()).real).sum() / w))
    out = []
    for i in range(S):
        for j in range(i + 1):
            for k in range(j + 1):
                nt = round(float((ones[i] * ones[j] * ones[k]).sum()) / float(N) ** 3)
                if nt:
                    noise = (mean[i] + mean[j] + mean[k] - 2 * b["S3"]) / b["I33"]
                    out.append((i, j, k, nt, float((fields[i] * fields[j] * fields[k]).sum()), noise))
    return out


# few shells, whose sums need the side given: 3 n_max + 1 = 100, 184, 364 and 472
@pytest.mark.parametrize("N,bs,side", [(128, (8, 8, 3, 4), 128), (200, (20, 20, 3, 3), 192), (384, (40, 40, 3, 3), 384),
                                       (512, (52, 52, 3, 3), 512)], ids=["128", "192", "384", "512"])
@pytest.mark.parametrize("contraction", [0, 2], ids=["fp32", "bf16x6"])
def test_shell_transforms(N, bs, side, contraction):
    """T_0 and the shot noise N_0 of every triangle against the FP64 transform
    of the same gridded fields."""
    import paper_1506_02729_gb300 as fkp
    n_max = math.ceil(bs[0] + (bs[3] - 1) * bs[1] + 0.5 * bs[2]) - 1
    assert 3 * n_max < side <= N
    sv = mockgen.survey_small(N=N, assign=3)
    gal, ran = mockgen.catalog(sv, 6)
    g, r = to_device(gal), to_device(ran)
    kf = 2 * math.pi / sv.L
    plan = fkp.Plan(sv.geometry(), (0.5 * kf, kf, 16), bshells=bs, want=1 | 16)
    b = plan.bispectrum(g, r, contraction=contraction)[1]
    F, Fw = (torch.from_numpy(a).cuda().double() * 2.0 ** -40 for a in plan.grid(g, r, with_w=True))
    ref = _monopole(F, Fw, bs, 3, b)
    assert [tuple(t) for t in b["tri"].astype(int)] == [t[:3] for t in ref]
    assert list(b["NT"]) == [t[3] for t in ref]
    T, noise = np.array([t[4] for t in ref]), np.array([t[5] for t in ref])
    assert np.max(np.abs(b["T0"] - T) / np.maximum(np.abs(T), np.median(np.abs(T)))) < B_TOL
    assert np.max(np.abs(b["N0"] - noise)) < SN_TOL * np.abs(noise).max()


@pytest.mark.parametrize("N", [128, 256, 384, 512])
def test_per_object_fields(N):
    """One line of sight for all objects (an observer at infinity, along no
    axis): the moment fields gridded per object are the node fields, and the
    spectra are the node plan's within the bound on either."""
    import paper_1506_02729_gb300 as fkp
    sv = mockgen.survey_small(N=N, assign=2)
    gal, ran = mockgen.catalog(sv, 7)
    g, r = to_device(gal), to_device(ran)
    geom = dict(sv.geometry(), observer=None, los=(1.0, 2.0, 2.0))
    kf = 2 * math.pi / sv.L
    want = fkp.FKP_P0 | fkp.FKP_P2 | fkp.FKP_P4 | fkp.FKP_P4B
    ref = fkp.Plan(geom, (0.5 * kf, kf, N // 2), want=want).power(g, r)
    got = fkp.Plan(geom, (0.5 * kf, kf, N // 2), want=want | fkp.FKP_XHAT_OBJECT).power(g, r)
    assert np.array_equal(got["nmodes"], ref["nmodes"])
    assert max(p_errors(got, ref).values()) < P_TOL, p_errors(got, ref)
