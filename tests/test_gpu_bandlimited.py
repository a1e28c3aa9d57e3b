"""Band-limited staging (blocks of frames staged as coefficients on the energies' band): segments of
512 frames and more, against the FP64 oracle at the suite's 1e-5 of the peak, at the sizes where the
blocks can go wrong: last blocks of 1 and of B - 1 frames, pushes that end inside blocks, pushes longer
and shorter than a block, rings of several flushes, ragged rows, each staging precision, energies of
either sign, uneven grids, FFT bins."""
import numpy as np
import pytest

import oracle
from synth import Detector, StreamSpec, frames
from tests.helpers import oracle_kw, rel_err_peak, run_gpu, stream_config

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_02236_gb300 import build
    build.build_all()


def spec_of(T, nw, E_max, K=12, **kw):
    return StreamSpec(P=3, Kx=K, Ky=K + 1, T=T, Tc=64, n_omega=nw, E_max_meV=E_max, n_modes=6, noise=1e-3,
                      detectors=(Detector(r_out=4.0),), **kw)


def cut(T, sizes):
    out, i = [], 0
    while sum(out) < T:
        out.append(min(sizes[i % len(sizes)], T - sum(out)))
        i += 1
    return out


# T, energies, E_max, push sizes, k_stage: E_max 60 / 120 / 150 / 250 meV give ranks from 8 to 48
CASES = [(513, 200, 120.0, [32], 0),           # a last block of one frame
         (575, 300, 120.0, [64], 0),           # ... of B - 1 frames (B = 64)
         (1000, 700, 150.0, [64, 64, 7, 121], 0),   # pushes that end inside blocks, and span two
         (640, 400, 250.0, [640], 0),          # the segment in one push
         (700, 260, 60.0, [20], 0),            # every block through the carry
         (1024, 300, 120.0, [32], 256),        # four flushes
         (1152, 500, 150.0, [128, 256], 384),  # three flushes, pushes across ring ends
         (2048, 130, 120.0, [8, 24], 0),
         # two-level sums: nine energy tiles, a last superblock of 33 frames, rings of two superblocks
         (2081, 950, 150.0, [64], 0),
         (4096, 1000, 150.0, [64, 128], 1024)]


@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_segments_against_the_oracle(case, precision):
    T, nw, E_max, sizes, k_stage = CASES[case]
    spec = spec_of(T, nw, E_max, subtract_mean=case % 3 != 1, window=("hann", "gauss", "rect")[case % 3])
    fr = frames.frames(spec, 40 + case, 0, T)
    out = run_gpu(spec, fr, precision, pushes=cut(T, sizes), k_stage=k_stage, want_psi=True)
    ref = oracle.forward(fr, **oracle_kw(spec))
    for name, want in (("I", ref.I), ("S", ref.S), ("Psi", ref.Psi)):
        e = rel_err_peak(out[name], want)
        assert e <= TOL, (name, e)
    if k_stage:
        assert out["info"]["flushes"] == -(-T // k_stage)


@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
@pytest.mark.parametrize("grid", ["signed", "offset", "uneven", "one", "fft"])
def test_energy_grids(grid, precision):
    """Bands about zero, away from zero (the elastic part outside the band, mean kept), uneven and
    unsorted energies, a single energy, few FFT bins."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    T = 768
    spec = spec_of(T, 150, 120.0, subtract_mean=grid != "offset")
    fr = frames.frames(spec, 7, 0, T)
    cfg, kw = stream_config(spec), oracle_kw(spec)
    rng = np.random.default_rng(3)
    E = {"signed": np.linspace(-60.0, 60.0, 150), "offset": np.linspace(40.0, 110.0, 150),
         "uneven": rng.permutation(120.0 * (np.arange(150) / 150.0) ** 2), "one": np.array([33.0]),
         "fft": None}[grid]
    if E is None:
        cfg.E_meV, cfg.fft_bins = None, 90
        kw.pop("E_meV")
        kw["fft_bins"] = 90
        nw = 90
    else:
        cfg.E_meV, kw["E_meV"], nw = [float(e) for e in E], E, len(E)
    buf = torch.from_numpy(np.ascontiguousarray(fr.transpose(1, 0, 2, 3))).cuda()
    fb = spec.P * spec.Kx * spec.Ky * 8
    ref = oracle.forward(fr, **kw)

    def error(**plan_kw):
        with TacawPlan([cfg], precision=precision, **plan_kw) as plan:
            I = torch.empty(plan.info()["I_elems"], device="cuda")
            for t in range(0, T, 64):
                plan.push(0, buf.data_ptr() + t * fb, 64)
            plan.finalize(I)
        return rel_err_peak(I.cpu().numpy().reshape(spec.P, nw, spec.Ky, spec.Kx), ref.I)

    e = error()
    if grid == "offset" and precision == "split_bf16":
        # an elastic line a hundred times the signal, outside the energies, in 16-bit pieces: the frames
        # form (16-frame rows) itself is 5.9e-5 off, so its error is the bound
        assert e <= error(tc_block_frames=16), e
    else:
        assert e <= TOL, e


def run_plan(cfgs, kw, bufs, pushes, grouped=False, state_at=None):
    """I and S of a plan pushed round-robin; state_at: also resumed in a second plan from that round."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan

    def rounds(plan, a, b):
        for r in range(a, b):
            todo = [(i, sum(p[:r]), p[r]) for i, p in enumerate(pushes) if r < len(p)]
            at = [bufs[i].data_ptr() + t * bufs[i].stride(0) * 8 for i, t, _ in todo]
            if grouped:
                plan.push_group([i for i, _, _ in todo], at, [n for _, _, n in todo])
            else:
                for (i, _, n), ptr in zip(todo, at):
                    plan.push(i, ptr, n)

    def done(plan):
        I = torch.zeros(plan.info()["I_elems"], device="cuda")
        S = torch.zeros(max(1, plan.info()["S_elems"]), device="cuda")
        plan.finalize(I, S)
        return I.cpu().numpy(), S.cpu().numpy()

    n = max(len(p) for p in pushes)
    with TacawPlan(cfgs, **kw) as plan:
        if state_at is None:
            rounds(plan, 0, n)
            return done(plan)
        rounds(plan, 0, state_at)
        state = plan.save_state()
    with TacawPlan(cfgs, **kw) as plan:
        plan.restore_state(state)
        rounds(plan, state_at, n)
        return done(plan) + (state,)


@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
def test_group_and_checkpoint_bit_identical(precision):
    """Three uneven streams (one of them short: frames staged as they are) with pushes that end inside
    blocks: group pushes, and a checkpoint with a partly filled block, give single pushes' bits."""
    import torch
    specs = [spec_of(640, 300, 120.0, K=10), spec_of(1100, 300, 120.0, K=14), spec_of(200, 90, 120.0, K=9)]
    frs = [frames.frames(s, 90 + i, 0, s.T) for i, s in enumerate(specs)]
    bufs = [torch.from_numpy(np.ascontiguousarray(f.transpose(1, 0, 2, 3))).cuda() for f in frs]
    cfgs = [stream_config(s) for s in specs]
    pushes = [cut(s.T, [48, 80]) for s in specs]
    kw = dict(precision=precision, k_stage=320, accum="kahan")
    ref = run_plan(cfgs, kw, bufs, pushes)
    got = run_plan(cfgs, kw, bufs, pushes, grouped=True)
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
    for cut_at in (3, 7):
        I, S, state = run_plan(cfgs, kw, bufs, pushes, state_at=cut_at)
        assert np.array_equal(ref[0], I) and np.array_equal(ref[1], S), cut_at
        # the staged coefficients are fewer than the frames they stand for
        staged = sum(8 * sum(p[:cut_at]) % (8 * 320) * ((s.P * s.Kx * s.Ky + 127) // 128 * 128)
                     for s, p in zip(specs[:2], pushes))
        acc = sum(16 * s.Nw * ((s.P * s.Kx * s.Ky + 127) // 128 * 128) for s in specs)
        assert state.size < 2 * (staged + acc)
    off = 0
    for s, fr in zip(specs, frs):
        n = s.P * s.Nw * s.Ky * s.Kx
        assert rel_err_peak(ref[0][off:off + n].reshape(s.P, s.Nw, s.Ky, s.Kx), oracle.forward(fr, **oracle_kw(s)).I) <= TOL
        off += n


def test_welch_lanes_and_pipelined_segments():
    """Overlapping Welch segments of 512 frames, and pipelined segments (bit-identical to unpipelined)."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    spec = spec_of(512, 200, 120.0, K=16)
    n = 40 + 2 * 256 + 512
    fr = frames.frames(spec_of(n, 200, 120.0, K=16), 5, 0, n)
    buf = torch.from_numpy(np.ascontiguousarray(fr.transpose(1, 0, 2, 3))).cuda()
    cfg = stream_config(spec)
    cfg.welch_segments, cfg.welch_stride, cfg.skip_init = 3, 256, 40
    ref = oracle.welch_forward(fr, 512, 256, skip_init=40, **oracle_kw(spec))
    for precision in ("split_bf16", "fp32"):
        I, S = run_plan([cfg], dict(precision=precision), [buf], [cut(n, [32])])
        assert rel_err_peak(I.reshape(ref.I.shape), ref.I) <= TOL
    cfg = stream_config(spec)
    st = torch.cuda.current_stream()
    outs = []
    for pipe in (False, True):
        with TacawPlan([cfg], precision="split_bf16") as plan:
            plan.set_pipelined_segments(pipe)
            Is = [torch.empty(plan.info()["I_elems"], device="cuda") for _ in range(2)]
            for k in range(2):
                plan.reset(st)
                for t in range(0, 512, 32):
                    plan.push(0, buf.data_ptr() + (k * 512 + t) * buf.stride(0) * 8, 32, st)
                plan.finalize_async(Is[k], None, None, st)
            if pipe:
                plan.drain(st)
            plan.check_errors(st)
            outs.append([I.cpu().numpy() for I in Is])
    for k in range(2):
        assert np.array_equal(outs[0][k], outs[1][k])
        ref = oracle.forward(fr[:, k * 512:(k + 1) * 512], **oracle_kw(spec))
        assert rel_err_peak(outs[0][k].reshape(ref.I.shape), ref.I) <= TOL
