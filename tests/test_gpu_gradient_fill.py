"""The spectrum's backward takes uninitialised memory for its gradient where the frames are the ROI alone and
zeros elsewhere: both against tacaw_backward into a cleared buffer, out of memory filled with NaN before.
(The same kernels run on the same inputs: 1e-5 of the peak leaves room for sums in another order.)"""
import math

import pytest

pytestmark = pytest.mark.gpu

CASES = {
    "roi": {},
    "one-probe": dict(n_probes=1, pitch_probe=1),
    "cropped": dict(gx=40, gy=36),
    "pitched-frames": dict(extra=64),
    "skipped": dict(skip_init=7),
    "welch-overlap": dict(welch_segments=3, welch_stride=40, skip_init=5),
    "welch-gap": dict(welch_segments=2, welch_stride=100),
}


@pytest.mark.parametrize("adjoint", ["split_bf16", "fp32"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_gradient_out_of_used_memory(name, adjoint):
    import torch
    from paper_2607_02236_gb300 import build
    from paper_2607_02236_gb300.autograd import spectrum
    from paper_2607_02236_gb300.tacaw import DetectorConfig, StreamConfig, TacawPlan
    build.build_all()
    kw = dict(CASES[name])
    kx, ky, T, nw = 27, 22, 80, 31
    gx, gy, P, extra = kw.pop("gx", kx), kw.pop("gy", ky), kw.pop("n_probes", 3), kw.pop("extra", 0)
    pitch_frame = P * gx * gy + extra
    cfg = StreamConfig(**{**dict(n_probes=P, kx=kx, ky=ky, T=T, dt_fs=5.0, pitch_row=gx, pitch_frame=pitch_frame,
                                 pitch_probe=gx * gy, roi_x0=(gx - kx) // 2, roi_y0=(gy - ky) // 2,
                                 E_meV=[3.0 * j for j in range(nw)], window="hann", subtract_mean=True,
                                 detectors=[DetectorConfig(kind="circular", r_out=6.0)]), **kw})
    n_seg = max(1, cfg.welch_segments)
    total = cfg.skip_init + (n_seg - 1) * (cfg.welch_stride or T) + T
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.polar(torch.rand(total * pitch_frame, device="cuda", generator=g),
                    2 * math.pi * torch.rand(total * pitch_frame, device="cuda", generator=g)).requires_grad_(True)
    c = torch.randn(P, 1, nw, device="cuda", generator=g)
    plan = TacawPlan([cfg], precision="fp32")
    plan.set_adjoint_precision(adjoint)
    S = spectrum(x, plan)
    want = torch.zeros_like(x)
    plan.backward(0, c, x.detach(), want, torch.cuda.current_stream())
    used = [torch.full_like(want, float("nan")) for _ in range(4)]
    del used                                    # the allocator hands these blocks to the backward
    (S * c).sum().backward()
    torch.cuda.synchronize()
    plan.close()
    assert torch.isfinite(torch.view_as_real(x.grad)).all()
    assert (x.grad - want).abs().max() <= 1e-5 * want.abs().max()
    assert torch.equal(x.grad == 0, want == 0)
