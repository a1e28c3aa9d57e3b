"""Band-limited staging where its forms are picked: rows enough for the rule to choose blocks of a known
length (read back from the plan's checkpoint, which records the form of each ring), pushes that leave
blocks unfinished, and plans whose segments change form.  Sampled pixels are held against the FP64
oracle at the suite's 1e-5 of the peak."""
import numpy as np
import pytest

import oracle
from tests.helpers import rel_err_peak

pytestmark = pytest.mark.gpu

TOL = 1e-5
KX, KY = 131, 127          # 16 637 rows: 3 of the last row tile's 128 are padding
ROWS = KX * KY


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_02236_gb300 import build
    build.build_all()


def config(T, nw, E_max, **kw):
    from paper_2607_02236_gb300 import DetectorConfig, StreamConfig
    base = dict(n_probes=1, kx=KX, ky=KY, T=T, dt_fs=5.0, pitch_row=KX, pitch_frame=ROWS, pitch_probe=ROWS,
                E_meV=list(np.arange(nw) * (E_max / nw)), detectors=[DetectorConfig(r_out=5.0)])
    base.update(kw)
    return StreamConfig(**base)


def waves(T, seed, E_max=120.0, elastic=1.0, rows=ROWS):
    """[T, rows] complex64 on the GPU: an elastic part, five lines inside the energies, noise."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.arange(T, device="cuda", dtype=torch.float64)
    E = E_max * (0.1 + 0.8 * torch.rand(5, device="cuda", dtype=torch.float64, generator=g))
    line = torch.exp(2j * np.pi * torch.frac(t[:, None] * (E * (5e-3 / 4.135667696)))).to(torch.complex64)
    amp = torch.polar(0.05 + 0.05 * torch.rand(5, rows, device="cuda", generator=g),
                      2 * np.pi * torch.rand(5, rows, device="cuda", generator=g))
    fr = line @ amp
    fr += elastic * torch.polar(torch.ones(rows, device="cuda"), 2 * np.pi * torch.rand(rows, device="cuda", generator=g))
    torch.view_as_real(fr).add_(torch.randn(T, rows, 2, device="cuda", generator=g), alpha=1e-4)
    return fr


def at(fr, t):
    return fr.data_ptr() + t * fr.stride(0) * 8


def push_all(plan, fr, sizes, a=0, b=None, push=None):
    """Frames [a, b) in pushes of the sizes in turn."""
    b = fr.shape[0] if b is None else b
    i = 0
    while a < b:
        n = min(sizes[i % len(sizes)], b - a)
        (push or plan.push)(0, at(fr, a), n)
        a += n
        i += 1


def ring_form(plan, stream=0):
    """Block length of the form the stream's ring holds (0: frames), from its checkpoint."""
    rec = plan.save_state()[48 + 48 * stream:48 + 48 * (stream + 1)]
    return int(rec[44:48].view(np.int32)[0])


def finish(plan, psi=False):
    """(I, Psi) [nw, rows] of the finished segment."""
    import torch
    n = plan.info()["I_elems"]
    I = torch.full((n,), -1.0, device="cuda")
    S = torch.empty(max(1, plan.info()["S_elems"]), device="cuda")
    P = torch.zeros(n, dtype=torch.complex64, device="cuda") if psi else None
    plan.finalize(I, S, P)
    return I.cpu().numpy().reshape(-1, ROWS), P.cpu().numpy().reshape(-1, ROWS) if psi else None


PIX = np.r_[0:16, 1000:16000:997, ROWS - 16:ROWS]


def assert_exact(I, fr, cfg, Psi=None):
    kw = dict(window_kind=cfg.window, window_param=cfg.window_param, E_meV=cfg.E_meV, fft_bins=cfg.fft_bins,
              subtract_mean=cfg.subtract_mean)
    psi, want = oracle.forward_pixels(fr[:, PIX].cpu().numpy(), **kw)
    e = rel_err_peak(I[:, PIX], want)
    assert e <= TOL, e
    if Psi is not None:
        e = rel_err_peak(Psi[:, PIX], psi)
        assert e <= TOL, e


@pytest.mark.parametrize("precision", ["split_fp16", "split_bf16"])
def test_unfinished_blocks_after_another_form(precision):
    """A segment of plain frames, then one of 16-frame pushes into blocks of 64: three of four pushes only
    carry, and the place of the carry holds the first segment's staged frames.  Rows past the last one take
    no part: no range error, and the results of a plan's first segment."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(1024, 1000, 150.0)
    fr = waves(1024, 3)
    with TacawPlan([cfg], precision=precision) as plan:
        push_all(plan, fr, [8])
        finish(plan)
        plan.reset()
        push_all(plan, fr, [16], 0, 48)
        assert ring_form(plan) == 64
        push_all(plan, fr, [16], 48)
        I, _ = finish(plan)
    assert_exact(I, fr, cfg)
    with TacawPlan([cfg], precision=precision) as plan:
        push_all(plan, fr, [16])
        assert np.array_equal(finish(plan)[0], I)


@pytest.mark.parametrize("nw,ring", [(1000, 64), (100, 0)])
def test_pipelined_plan_single_and_group_pushes(nw, ring):
    """A pipelined plan takes single and group pushes of one segment: the first segment's converted at push
    time (into blocks of 64 frames at 1000 energies, as plain frames at 100), the second's while the first's
    contraction is pending.  The bits are those of an unpipelined plan's single pushes."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(1024, nw, 150.0)
    frs = [waves(1024, 5), waves(1024, 6)]
    st = torch.cuda.current_stream()
    outs = []
    for pipe in (False, True):
        with TacawPlan([cfg], precision="split_bf16") as plan:
            plan.set_pipelined_segments(pipe)
            Is = [torch.full((plan.info()["I_elems"],), -1.0, device="cuda") for _ in frs]
            for k, fr in enumerate(frs):
                plan.reset(st)
                for i, t in enumerate(range(0, 1024, 32)):
                    if pipe and i % 3:
                        plan.push_group([0], [at(fr, t)], [32], st)
                    else:
                        plan.push(0, at(fr, t), 32, st)
                    if k == 0 and i == 1:
                        assert ring_form(plan) == ring
                plan.finalize_async(Is[k], None, None, st)
            if pipe:
                plan.drain(st)
            plan.check_errors(st)
            outs.append([I.cpu().numpy().reshape(-1, ROWS) for I in Is])
    for k, fr in enumerate(frs):
        assert np.array_equal(outs[0][k], outs[1][k])
        assert_exact(outs[0][k], fr, cfg)


def no_room(cfg, k_stage, **kw):
    """Plan arguments whose budget is what the plan needs without any form's tables."""
    import re
    from paper_2607_02236_gb300 import TacawError, TacawPlan
    with pytest.raises(TacawError) as e:
        TacawPlan([cfg], k_stage=k_stage, hbm_budget_bytes=1, **kw)
    return dict(kw, k_stage=k_stage, hbm_budget_bytes=int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)))


@pytest.mark.parametrize("mean", [False, True])
@pytest.mark.parametrize("ring,sizes", [(0, [8]), (64, [64, 16])])
@pytest.mark.parametrize("saver", ["with forms", "without"])
def test_checkpoint_between_plans_with_and_without_forms(saver, ring, sizes, mean):
    """A plan with memory for band-limited forms and one without take each other's checkpoints, also where the
    stream keeps its mean (which a plan with forms takes out of the frames and adds back) and where the ring
    holds coefficients (the loader then builds that form's tables)."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(1024, 1000, 150.0, subtract_mean=mean)
    fr = waves(1024, 8)
    plans = [dict(precision="split_bf16", k_stage=1024), no_room(cfg, 1024, precision="split_bf16")]
    if saver == "without":
        plans.reverse()
    with TacawPlan([cfg], **plans[0]) as A:
        push_all(A, fr, sizes, 0, 144)
        assert ring_form(A) == (ring if saver == "with forms" else 0)
        state = A.save_state()
    with TacawPlan([cfg], **plans[1]) as B:
        push_all(B, fr, [64], 0, 64)          # a segment in progress that the checkpoint replaces
        assert ring_form(B) == (0 if saver == "with forms" else 64)
        B.restore_state(state)
        push_all(B, fr, [64], 144)
        I, _ = finish(B)
    assert_exact(I, fr, cfg)


def test_checkpoint_versions():
    """Checkpoints of the version before forms (plain frames, kept mean left in them) are read; later ones not."""
    from paper_2607_02236_gb300 import TacawError, TacawPlan
    cfg = config(256, 64, 120.0)
    fr = waves(256, 9)
    with TacawPlan([cfg], precision="split_bf16") as plan:
        push_all(plan, fr, [32], 0, 96)
        state = plan.save_state()
        push_all(plan, fr, [32], 96)
        want, _ = finish(plan)
        version = int(state[8:12].view(np.uint32)[0])
        assert version == 2
        for v, ok in ((1, True), (2, True), (3, False), (0, False)):
            state[8:12] = np.frombuffer(np.uint32(v).tobytes(), np.uint8)
            if not ok:
                with pytest.raises(TacawError, match="version"):
                    plan.restore_state(state)
                continue
            plan.restore_state(state)
            push_all(plan, fr, [32], 96)
            assert np.array_equal(finish(plan)[0], want)


def row_scales(plan):
    """Scales of the rows' staged coefficients (the last section of a checkpoint between blocks)."""
    return plan.save_state()[-4 * (-(-ROWS // 128) * 128):].copy().view(np.float32)


@pytest.mark.parametrize("precision", ["split_bf16", "split_fp16"])
def test_windows_that_start_low_keep_their_rows_scale(precision):
    """Blackman-Harris grows by 2^14 from a segment's first block to its middle: the rows' scales, set with the
    first block, take that into account and hold to the end."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(2048, 400, 120.0, window="blackmanharris")
    fr = waves(2048, 13)
    with TacawPlan([cfg], precision=precision) as plan:
        push_all(plan, fr, [64], 0, 64)
        assert ring_form(plan) == 64
        first = row_scales(plan)
        push_all(plan, fr, [64], 64)
        assert np.array_equal(row_scales(plan), first)
        I, Psi = finish(plan, psi=True)
    assert_exact(I, fr, cfg, Psi)


@pytest.mark.parametrize("precision,T,sizes,ring", [("split_bf16", 1024, [64], 64), ("split_fp16", 1024, [64], 64),
                                                    ("split_bf16", 2048, [32], 32), ("split_bf16", 1024, [48], 64)])
def test_rows_that_outgrow_their_scale(precision, T, sizes, ring):
    """Bursts of 2^12 to 2^24 times the earlier signal, in a third of the rows and at places that differ from row
    to row, have the staged coefficients of those rows rescaled, some of them twice."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(T, 1000 if ring == 64 else 400, 150.0 if ring == 64 else 120.0, window="rect")
    fr = waves(T, 14, elastic=0.0) * 1e-4
    g = torch.Generator(device="cuda").manual_seed(15)
    row = torch.arange(ROWS, device="cuda")
    for factor, a, b in ((2.0 ** 12, T // 8, T // 2), (2.0 ** 12, T // 2, 7 * T // 8)):
        at_row = torch.randint(a, b, (ROWS,), device="cuda", generator=g)
        at_row = torch.where(row % 3 == 1, at_row, T)
        fr *= torch.where(torch.arange(T, device="cuda")[:, None] >= at_row[None, :], factor, 1.0)
    with TacawPlan([cfg], precision=precision, **({"fp16_scale": 16.0} if precision == "split_fp16" else {})) as plan:
        push_all(plan, fr, sizes, 0, sizes[0])
        first = None
        if sizes[0] == ring:
            assert ring_form(plan) == ring
            first = row_scales(plan)
        push_all(plan, fr, sizes, sizes[0])
        if first is not None:
            changed = (row_scales(plan) != first)[:ROWS]
            assert changed[1::3].all() and not changed[0::3].any()
        I, Psi = finish(plan, psi=True)
    # rows of very different size: each against its own peak
    kw = dict(window_kind="rect", E_meV=cfg.E_meV)
    psi, want = oracle.forward_pixels(fr[:, PIX].cpu().numpy(), **kw)
    for k, p in enumerate(PIX):
        assert rel_err_peak(I[:, p], want[:, k]) <= TOL, (p, p % 3)
        assert rel_err_peak(Psi[:, p], psi[:, k]) <= TOL, (p, p % 3)


@pytest.mark.parametrize("precision", ["split_bf16", "split_fp16"])
def test_accumulators_of_rings_in_a_far_tail(precision):
    """Four flushes under a Gauss window whose first and last rings hold 1e-38 of its maximum: their rows are
    scaled up by as much as 2^120, where the plain FP32 accumulators of the rings before have no place."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(2048, 1000, 150.0, window="gauss", window_param=38.8)
    fr = waves(2048, 17) * 1e3
    with TacawPlan([cfg], precision=precision, k_stage=512, accum="fp32",
                   **({"fp16_scale": 4.0} if precision == "split_fp16" else {})) as plan:
        push_all(plan, fr, [64], 0, 1600)
        assert ring_form(plan) == 64
        push_all(plan, fr, [64], 1600)
        I, Psi = finish(plan, psi=True)
        assert plan.info()["flushes"] == 4
    assert_exact(I, fr, cfg, Psi)


@pytest.mark.parametrize("precision,ring,sizes", [("fp32", 128, [128]), ("fp32", 128, [200, 56]), ("fp32", 128, [16]),
                                                  ("split_bf16", 64, [64]), ("split_bf16", 64, [16]),
                                                  ("split_fp16", 64, [100, 28])])
def test_residual_sums_are_exact_to_a_few_frames(precision, ring, sizes):
    """The sums behind the exact mean run in FP32 over 8 frames (FP32 path) or 32 (split path) and are exact from
    there on: frames of 1 + 2^-20 (2^-19) sum without a rounding up to 8 (32) of them, and lose bits in longer
    FP32 sums.  The first 32 frames, which give the provisional mean, are zero."""
    from paper_2607_02236_gb300 import TacawPlan
    T = 1024
    cfg = config(T, 1000, 150.0)
    fr = waves(T, 11, elastic=0.0) * 0
    one = 1 + 2.0 ** (-20 if precision == "fp32" else -19)
    fr[32:] = one * (1 - 1j)
    with TacawPlan([cfg], precision=precision) as plan:
        push_all(plan, fr, [32] if sizes == [16] else sizes, 0, 32 if sizes == [16] else sizes[0])
        a = 32 if sizes == [16] else sizes[0]
        push_all(plan, fr, sizes, a, 768)
        assert ring_form(plan) == ring
        state = plan.save_state()
    off = 48 + 48 + 8 + 8 * ROWS           # behind the header, the counters and the provisional means
    sums = state[off:off + 16 * ROWS].copy().view(np.complex128)
    assert np.all(sums == (768 - 32) * one * (1 - 1j))


@pytest.mark.parametrize("nw,sizes,ring", [(400, [32], 32), (1000, [64], 64)])
def test_split_fp16_kept_mean_outside_the_energies(nw, sizes, ring):
    """A kept elastic line 300 times the signal, 20 meV below the energies: it is taken out of the frames before
    they become coefficients, whose 22 bits would otherwise be spent on it."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(2048, nw, 100.0, window="rect", subtract_mean=False, E_meV=list(20.0 + np.arange(nw) * (100.0 / nw)))
    fr = waves(2048, 19, elastic=30.0)
    with TacawPlan([cfg], precision="split_fp16", fp16_scale=1024.0) as plan:
        push_all(plan, fr, sizes, 0, 256)
        assert ring_form(plan) == ring
        push_all(plan, fr, sizes, 256)
        I, Psi = finish(plan, psi=True)
    assert_exact(I, fr, cfg, Psi)


@pytest.mark.parametrize("first,ring", [(64, 64), (8, 0)])
def test_split_fp16_kept_mean_range(first, ring):
    """Frames that change sign after the first 32, at 0.94 of the fp16 range: accepted, with residuals beyond the
    range, in a segment of two rings that both take the first one's kind of form.  Beyond the range: refused."""
    from paper_2607_02236_gb300 import TacawError, TacawPlan
    cfg = config(1024, 1000, 150.0, subtract_mean=False)
    fr = waves(1024, 21, elastic=0.0) * 0.1
    fr[:32] += 15 - 15j
    fr[32:] -= 15 - 15j
    with TacawPlan([cfg], precision="split_fp16", k_stage=512) as plan:
        push_all(plan, fr, [first], 0, 512)
        push_all(plan, fr, [8 if ring else 64], 512, 576)
        assert (ring_form(plan) > 0) == (ring > 0)
        state = plan.save_state()
        push_all(plan, fr, [64], 576)
        I, _ = finish(plan)
        if ring:
            assert_exact(I, fr, cfg)
        plan.restore_state(state)
        push_all(plan, fr, [64], 576)
        assert np.array_equal(finish(plan)[0], I)
        for t in (1, 500, 1000):
            plan.reset()
            bad = fr[t].clone()
            fr[t, 7] = 16.1
            with pytest.raises(TacawError, match="fp16 range"):
                push_all(plan, fr, [first])
                finish(plan)
            fr[t] = bad
            plan.close()
            plan.__init__([cfg], precision="split_fp16", k_stage=512)


def device_bytes(cfg, **kw):
    from paper_2607_02236_gb300 import TacawPlan
    with TacawPlan([cfg], **kw) as plan:
        return plan.info()["device_bytes"]


def test_tables_only_for_forms_a_push_can_take_and_once_a_stream():
    """Few rows: no push length makes a form worth its launches, so none is built.  The lanes of a Welch average
    share one set of tables."""
    kw = dict(precision="split_bf16")
    small = config(1024, 60, 120.0, kx=36, ky=13, pitch_row=36, pitch_frame=468, pitch_probe=468)
    assert device_bytes(small, k_stage=1024, **kw) == device_bytes(small, **no_room(small, 1024, **kw))
    tables = []
    for stride in (256, 128):               # 2 and 4 lanes
        cfg = config(512, 1000, 150.0, welch_segments=5, welch_stride=stride)
        tables.append(device_bytes(cfg, k_stage=512, **kw) - device_bytes(cfg, **no_room(cfg, 512, **kw)))
    assert tables[0] == tables[1] > 0


@pytest.mark.parametrize("precision", ["split_bf16", "split_fp16", "fp32"])
@pytest.mark.parametrize("mean", [True, False])
def test_welch_lanes_in_blocks(precision, mean):
    """Overlapping Welch segments that take the form, pushes of whole blocks of every lane."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(512, 1000, 150.0, welch_segments=3, welch_stride=256, subtract_mean=mean)
    n = 2 * 256 + 512
    fr = waves(n, 23)
    with TacawPlan([cfg], precision=precision) as plan:
        push_all(plan, fr, [64], 0, 320)
        B = 128 if precision == "fp32" else 64
        assert [ring_form(plan, i) for i in range(2)] == [B, B]
        state = plan.save_state()
        push_all(plan, fr, [64], 320)
        I, _ = finish(plan)
    with TacawPlan([cfg], **no_room(cfg, 512, precision=precision)) as plan:
        plan.restore_state(state)           # builds the lanes' tables
        push_all(plan, fr, [64], 320)
        assert rel_err_peak(finish(plan)[0], I) <= TOL
    ref = oracle.welch_forward(fr[:, PIX].cpu().numpy()[None, :, None, :], 512, 256, E_meV=cfg.E_meV, subtract_mean=mean)
    assert rel_err_peak(I[:, PIX], ref.I[0, :, 0]) <= TOL


def test_a_push_across_a_ring_end_keeps_the_form():
    """Pushes of 96 frames into rings of 512: the second ring begins with 64 frames of one.  Its form is that of pushes
    of 96 (blocks of 32), not of 64 (blocks of 64), into which every later push would end."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(1024, 600, 150.0)
    fr = waves(1024, 25)
    with TacawPlan([cfg], precision="split_bf16", k_stage=512) as plan:
        push_all(plan, fr, [96], 0, 96)
        assert ring_form(plan) == 32
        push_all(plan, fr, [96], 96, 576)
        assert ring_form(plan) == 32
        push_all(plan, fr, [96], 576)
        I, _ = finish(plan)
        assert_exact(I, fr, cfg)
        plan.reset()
        push_all(plan, fr, [64], 0, 64)
        assert ring_form(plan) == 64


PRECISIONS = ["split_bf16", "split_fp16", "fp32"]

# T, energies, E_max, push sizes, k_stage, accumulators, block length on the split and on the FP32 path
CASES = [(1000, 1000, 150.0, [64], 0, "auto", 64, 128),             # a last block of 40 (104) frames
         (1025, 1000, 150.0, [64], 0, "auto", 64, 128),             # ... of one frame
         (1023, 1000, 150.0, [100, 28], 0, "auto", 64, 128),        # ... of all but one; pushes that end inside blocks
         (1000, 1000, 150.0, [63, 65, 1], 0, "auto", 64, 128),      # chunks of four frames parted
         (1000, 1000, 150.0, [16], 0, "auto", 64, 128),             # three of four pushes only carry
         (2081, 400, 120.0, [32], 0, "auto", 32, 128),              # split: two levels, a last superblock of 33 frames
         (2081, 1000, 150.0, [64], 0, "auto", 64, 128),             # split: two levels, superblocks of 512
         (1000, 700, 60.0, [64], 0, "auto", 64, 128),               # small ranks, two levels
         (1024, 1000, 240.0, [64], 0, "auto", 64, 64),              # the greatest rank of the split path
         (2048, 1000, 150.0, [64], 512, "kahan", 64, 128),          # four flushes
         (2048, 400, 120.0, [32], 512, "fp32", 32, 128),
         (1152, 1000, 150.0, [96], 384, "fp64", 64, 128)]           # pushes across the rings' ends


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("case", range(len(CASES)))
def test_forms_against_the_oracle(case, precision):
    from paper_2607_02236_gb300 import TacawPlan
    T, nw, E_max, sizes, k_stage, accum, split, fp32 = CASES[case]
    cfg = config(T, nw, E_max, window=("hann", "gauss", "rect")[case % 3], window_param=T / 6.0 if case % 3 == 1 else 0.0,
                 subtract_mean=case % 4 != 1)
    fr = waves(T, 30 + case)
    with TacawPlan([cfg], precision=precision, k_stage=k_stage, accum=accum) as plan:
        push_all(plan, fr, sizes, 0, sizes[0])
        assert ring_form(plan) == (fp32 if precision == "fp32" else split)
        push_all(plan, fr, sizes[1:] + sizes[:1], sizes[0])
        I, Psi = finish(plan, psi=True)
        if k_stage:
            assert plan.info()["flushes"] == -(-T // k_stage)
    assert_exact(I, fr, cfg, Psi)


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("grid", ["signed", "uneven", "offset", "fft"])
def test_energy_grids_in_blocks(grid, precision):
    from paper_2607_02236_gb300 import TacawPlan
    T = 4000 if grid == "fft" else 768
    rng = np.random.default_rng(3)
    E = {"signed": np.linspace(-90.0, 90.0, 600), "uneven": rng.permutation(120.0 * (np.arange(600) / 600.0) ** 2),
         "offset": np.linspace(40.0, 160.0, 600), "fft": None}[grid]
    cfg = config(T, 600, 120.0, subtract_mean=grid != "offset")
    cfg.E_meV, cfg.fft_bins = (None, 900) if E is None else ([float(e) for e in E], 0)
    fr = waves(T, 40)
    with TacawPlan([cfg], precision=precision) as plan:
        push_all(plan, fr, [64], 0, 64)
        assert ring_form(plan) == (128 if precision == "fp32" else 64)
        push_all(plan, fr, [64], 64)
        I, Psi = finish(plan, psi=True)
    assert_exact(I, fr, cfg, Psi)


@pytest.mark.parametrize("precision", PRECISIONS)
def test_groups_and_checkpoints_of_streams_in_blocks(precision):
    """Two streams of different length, pushes that end inside blocks, two rings a segment: group pushes and a
    checkpoint with unfinished blocks give the bits of single pushes, and the checkpoint is smaller than the frames
    it stands for."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    cfgs = [config(1024, 1000, 150.0), config(768, 1000, 150.0, subtract_mean=False)]    # rings of 512 and 384
    frs = [waves(1024, 51), waves(768, 52)]
    sizes = [48, 80]

    def rounds(plan, a, b, grouped):
        done = [0, 0]
        for r in range(b):
            todo = [(i, done[i], min(sizes[r % 2], c.T - done[i])) for i, c in enumerate(cfgs) if done[i] < c.T]
            for i, _, n in todo:
                done[i] += n
            if r < a:
                continue
            if grouped:
                plan.push_group([i for i, _, _ in todo], [at(frs[i], t) for i, t, _ in todo], [n for _, _, n in todo])
            else:
                for i, t, n in todo:
                    plan.push(i, at(frs[i], t), n)
        return done

    def outputs(plan):
        I = torch.zeros(plan.info()["I_elems"], device="cuda")
        plan.finalize(I)
        return I.cpu().numpy().reshape(2, -1, ROWS)

    kw = dict(precision=precision, k_stage=512, accum="kahan")
    with TacawPlan(cfgs, **kw) as plan:
        rounds(plan, 0, 16, False)
        ref = outputs(plan)
        plan.reset()
        rounds(plan, 0, 16, True)
        assert np.array_equal(outputs(plan), ref)
        for cut_at in (3, 5, 9):            # 176, 304 (in the first rings) and 560 frames
            plan.reset()
            done = rounds(plan, 0, cut_at, True)
            state = plan.save_state()
            B = 128 if precision == "fp32" else 64
            assert [ring_form(plan, i) for i in range(2)] == [B, B]
            pad = -(-ROWS // 128) * 128
            if cut_at < 9:
                assert state.size < sum(24 * ROWS + 8 * d * pad for d in done)
            with TacawPlan(cfgs, **kw) as other:
                other.restore_state(state)
                rounds(other, cut_at, 16, False)
                assert np.array_equal(outputs(other), ref)
    for i, (cfg, fr) in enumerate(zip(cfgs, frs)):
        assert_exact(ref[i], fr, cfg)


@pytest.mark.parametrize("precision", PRECISIONS)
def test_captured_segment_in_blocks(precision):
    """A segment in blocks captured into a graph: replays on new frames give the bits of eager passes."""
    import torch
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(2081, 400, 120.0, subtract_mean=False)
    frs = [waves(2081, 61), waves(2081, 62)]
    buf = frs[0].clone()
    st = torch.cuda.Stream()
    with TacawPlan([cfg], precision=precision) as plan:
        I = torch.zeros(plan.info()["I_elems"], device="cuda")

        def segment():
            plan.reset(st)
            for t in range(0, 2081, 32):
                plan.push(0, at(buf, t), min(32, 2081 - t), st)
            plan.finalize_async(I, None, None, st)

        want = []
        for fr in frs:
            buf.copy_(fr)
            torch.cuda.synchronize()
            segment()
            plan.check_errors(st)
            want.append(I.cpu().numpy().copy())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            segment()
        for k in (1, 0, 1):
            buf.copy_(frs[k])
            I.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(I.cpu().numpy(), want[k])
    assert_exact(want[1].reshape(-1, ROWS), frs[1], cfg)


def test_split_fp16_welch_segments_of_both_kinds():
    """A lane's first segment in blocks, its kept mean taken out, the next one as plain frames of the other sign at
    0.92 of the fp16 range: nothing of the first one's mean is left in the second's conversion."""
    from paper_2607_02236_gb300 import TacawPlan
    cfg = config(512, 1000, 150.0, subtract_mean=False, welch_segments=2, welch_stride=512)
    fr = waves(1024, 27, elastic=0.0)
    fr[:512] += 14.7
    fr[512:] -= 14.7
    with TacawPlan([cfg], precision="split_fp16") as plan:
        push_all(plan, fr, [64], 0, 64)
        assert ring_form(plan) == 64
        push_all(plan, fr, [64], 64, 512)
        push_all(plan, fr, [8], 512, 520)
        assert ring_form(plan) == 0
        push_all(plan, fr, [8], 520)
        I, _ = finish(plan)
    ref = oracle.welch_forward(fr[:, PIX].cpu().numpy()[None, :, None, :], 512, 512, E_meV=cfg.E_meV, subtract_mean=False)
    assert rel_err_peak(I[:, PIX], ref.I[0, :, 0]) <= TOL
