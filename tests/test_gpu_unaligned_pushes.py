"""Pushes that start and end inside the staged rows' 16-byte chunks (4 frames) and inside blocks of 16 and 32
frames, on every staged precision: the frames land where one push of the whole segment puts them (bit-identical
intensities with the mean kept), and match the FP64 oracle at the suite's 1e-5 of the peak with it removed."""
import numpy as np
import pytest

import oracle
from synth import Detector, StreamSpec, frames
from tests.helpers import oracle_kw, rel_err_peak, run_gpu

pytestmark = pytest.mark.gpu

TOL = 1e-5
PUSHES = {"ones": [1] * 9 + [23, 64, 64], "odd": [3, 7, 25, 31, 33, 6, 5, 17, 1, 32], "long": [1, 159], "chunks": [2, 4, 30, 60, 64]}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_02236_gb300 import build
    build.build_all()


@pytest.mark.parametrize("precision,kw", [("split_bf16", {}), ("split_bf16", dict(tc_block_frames=16)),
                                          ("split_bf16", dict(k_stage=64)), ("split_fp16", {}), ("fp32", {})])
@pytest.mark.parametrize("name", sorted(PUSHES))
def test_unaligned_pushes(name, precision, kw):
    base = dict(P=3, Kx=11, Ky=13, T=160, Tc=160, n_omega=60, E_max_meV=120.0, n_modes=6, noise=1e-3,
                detectors=(Detector(r_out=4.0),))
    kept = StreamSpec(subtract_mean=False, **base)
    fr = frames.frames(kept, 3, 0, kept.T)
    whole = run_gpu(kept, fr, precision, pushes=[160], **kw)
    parts = run_gpu(kept, fr, precision, pushes=PUSHES[name], **kw)
    assert np.array_equal(whole["I"], parts["I"])
    spec = StreamSpec(**base)
    out = run_gpu(spec, fr, precision, pushes=PUSHES[name], **kw)
    ref = oracle.forward(fr, **oracle_kw(spec))
    assert rel_err_peak(out["I"], ref.I) <= TOL
    assert rel_err_peak(out["S"], ref.S) <= TOL
