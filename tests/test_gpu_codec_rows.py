"""The encoder's and decoder's patch maps at every unit width: pieces of p v
values that 8, 4 or neither divides, channel counts that 4 divides or not,
levels padded or not, and fields that are not 16-byte aligned (bit for bit the
same result), against the FP64 oracle (FP32 1e-5, BF16 2e-2)."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm
import synth
from oracle import wm_oracle as orc

pytestmark = pytest.mark.gpu

BASE = dataclasses.replace(synth.SMALL_CODEC, Ce=128, heads=4, blocks=1, kd=1, kh=3, kw=3)
CASES = {
    "unit8": dataclasses.replace(BASE, H0=48, W0=72, p=8, levels=10, level_pad=12, pd=4),
    "unit4": dataclasses.replace(BASE, H0=20, W0=36, p=4, levels=7, level_pad=8, pd=2, v_sfc_out=5, n_const=4),
    "one_level": dataclasses.replace(BASE, H0=24, W0=40, p=8, levels=1, level_pad=1, pd=1, v_atm=3, v_sfc_in=4),
    "scalar": dataclasses.replace(BASE, H0=15, W0=21, p=3, levels=5, level_pad=6, pd=3, v_atm=5, n_const=3),
    "no_constants": dataclasses.replace(BASE, H0=16, W0=32, p=4, levels=4, level_pad=4, pd=2, n_const=0),
}


def _off(a, shift):
    """A device copy that starts `shift` floats past a 16-byte boundary."""
    a = np.ascontiguousarray(a, dtype=np.float32)
    buf = torch.empty(a.size + 4, device="cuda")
    t = buf[shift:shift + a.size].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("prec", [wm.WM_PREC_FP32, wm.WM_PREC_BF16])
@pytest.mark.parametrize("name", list(CASES))
def test_patch_units(name, prec):
    cd, C = CASES[name], 64
    if prec == wm.WM_PREC_BF16 and name == "scalar":
        pytest.skip("patch widths the BF16 codec does not take")
    w = synth.codec_weights(cd, C, seed=0, stress=True)
    atm, sfc, cst = synth.codec_inputs(cd, seed=1)
    tol = 1e-5 if prec == wm.WM_PREC_FP32 else 2e-2
    codec = wm.wm_codec_create(wm.make_codec_config(cd, C, prec), synth.pack_codec_weights(w))
    try:
        got = []
        for shift in (0, 1):
            lat = torch.empty(cd.D, cd.H, cd.W, C, device="cuda")
            wm.wm_encode(codec, _off(atm, shift), _off(sfc, shift), _off(cst, shift), lat)
            a_out = _off(np.full((cd.levels, cd.H0, cd.W0, cd.v_atm), np.nan), shift)
            s_out = _off(np.full((cd.H0, cd.W0, cd.v_sfc_out), np.nan), shift)
            wm.wm_decode(codec, lat, a_out, s_out)
            torch.cuda.synchronize()
            got.append([t.cpu().numpy() for t in (lat, a_out, s_out)])
        for a, b in zip(*got):
            assert np.array_equal(a, b)
        ref = orc.encode(atm, sfc, cst, w, cd)
        assert orc.rel_l2(got[0][0], ref) <= tol
        ra, rs = orc.decode(got[0][0], w, cd)
        assert orc.rel_l2(got[0][1], ra) <= tol and orc.rel_l2(got[0][2], rs) <= tol
    finally:
        wm.wm_codec_destroy(codec)
