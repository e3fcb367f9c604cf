"""The packer finds a weight's level through a table of bins: values on and beside every threshold and every bin edge, and
codebooks that share a bin or reach beyond the outermost, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, _np, _status_ok, dq  # noqa: F401

pytestmark = pytest.mark.gpu

CODEBOOKS = {
    "default": None,
    "one threshold per bin, barely": (-1.6, -1.0, -0.5, 0, 0.55, 1.1, 1.7, 6),
    "two in a bin": (-0.3, -0.2, -0.1, 0, 0.1, 0.2, 0.3, 6),
    "one far below the bins": (-300, -3, -1.5, 0, 1, 2.25, 4, 6),
    "two below the bins": (-300, -80, -20, 0, 1, 2.25, 4, 6),
    "threshold 0.95e-3 below a bin edge": (-4.703125, -2.869140625, -1.369140625, 0, 0.07489013671875, 2.462890625, 4.046875, 6),
    "threshold 0.97e-3 below a bin edge": (-4.703125, -3.5, -2.470703125, -0.0709228515625, 0, 2.5, 4, 6),
    "subnormal levels": (-3, -2, -2.0 ** -24, 0, 2.0 ** -24, 2, 4, 6),
}


def _codebook(oracle, name):
    return None if CODEBOOKS[name] is None else np.array([oracle.f16_encode(v) for v in CODEBOOKS[name]], dtype=np.uint16)


@pytest.mark.parametrize("name", list(CODEBOOKS))
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_pack_at_thresholds_and_bin_edges(dq, oracle, name, dtype):  # noqa: F811
    cb = _codebook(oracle, name)
    G = oracle.codebook_values(oracle.lut3_default_codebook() if cb is None else cb).astype(np.float32)
    T = (G[1:] + G[:-1]) * np.float32(0.5)
    edges = ((np.arange(64, dtype=np.float64) / 63 - 0.5) * 32).astype(np.float32)
    v = np.concatenate([T, edges, np.linspace(-6, 6, 97, dtype=np.float32), G, [0.0, -0.0]]).astype(np.float32)
    v = np.concatenate([v, np.nextafter(v, np.float32(-100)), np.nextafter(v, np.float32(100))])
    v = v[np.abs(v) < 6]
    # tensor scale 1 (largest magnitude 2688), block scales 1 (extreme 6 or -6): a weight is its own normalised value
    N, K = 48, 640
    W = np.zeros((N, K), np.float32)
    W[0, 0] = 2688
    blocks = W[1:].reshape(-1, 16)
    blocks[:, 1:] = np.resize(v, (blocks.shape[0], 15))
    blocks[:, 0] = np.where(np.arange(blocks.shape[0]) // (len(v) // 15 + 1) % 2 == 0, 6.0, -6.0)
    Wt = torch.from_numpy(W).to(dtype)
    ref = oracle.pack_weights(Wt.float().numpy(), cb)
    assert ref["s"] == 1.0
    w = dq.pack_weights(Wt.to(DEV), codebook_f16=cb)
    planes, lsc, _ = dq.export_canonical(w, dq.FMT_LUT3)
    codes, sc, _ = dq.export_canonical(w, dq.FMT_NVFP4)
    _status_ok(dq)
    assert np.array_equal(_np(lsc), ref["lut3_scales"]) and np.array_equal(_np(planes).view(np.uint32), ref["lut3_planes"])
    assert np.array_equal(_np(sc), ref["nvfp4_scales"]) and np.array_equal(_np(codes), ref["nvfp4_codes"])


@pytest.mark.parametrize("fmts", ["lut2", "nvfp4+lut2"])
def test_pack_lut2_at_thresholds(dq, oracle, fmts):  # noqa: F811
    G = oracle.codebook_values(oracle.lut2_default_codebook()).astype(np.float32)
    v = np.concatenate([(G[1:] + G[:-1]) * np.float32(0.5), np.linspace(-5.9, 5.9, 61, dtype=np.float32)])
    v = np.concatenate([v, np.nextafter(v, np.float32(-100)), np.nextafter(v, np.float32(100))])
    W = np.zeros((16, 1152), np.float32)
    W[0, 0] = 2688
    blocks = W[1:].reshape(-1, 16)
    blocks[:, 1:] = np.resize(v, (blocks.shape[0], 15))
    blocks[:, 0] = np.where(np.arange(blocks.shape[0]) % 3 == 0, -6.0, 6.0)
    w = dq.pack_weights(torch.from_numpy(W).to(DEV), formats=dq.FMT_LUT2 | (dq.FMT_NVFP4 if "nvfp4" in fmts else 0))
    planes, sc, _ = dq.export_canonical(w, dq.FMT_LUT2)
    _status_ok(dq)
    p, s = oracle.quant_lut2(W, 1.0)
    assert np.array_equal(_np(sc), s) and np.array_equal(_np(planes).view(np.uint32), p)


@pytest.mark.parametrize("kind", ["nan", "nan blocks", "one nan at the end", "infinity", "subnormal", "zero times a reciprocal beyond fp32"])
@pytest.mark.parametrize("N,K", [(48, 640), (272, 1152)])
def test_pack_encodings_do_not_depend_on_their_company(dq, kind, N, K):  # noqa: F811
    """An encoding has the same bytes whatever else is packed with it, and from fp32 as from bf16, also beside NaN, infinities and zeros that a
    reciprocal beyond fp32 turns into NaN: their E2M1 code has no sign that a negative block scale could turn round."""
    g = torch.Generator(device=DEV).manual_seed(N)
    W = torch.randn(N, K, generator=g, device=DEV) * 0.02
    blocks = W.view(-1, 16)
    if kind == "nan":
        W.view(-1)[torch.randperm(N * K, generator=g, device=DEV)[:N * K // 50]] = float("nan")
    elif kind == "nan blocks":
        blocks[::7], blocks[3::11, 5] = float("nan"), float("nan")
    elif kind == "one nan at the end":
        blocks[-1, 15], blocks[-1, 3] = float("nan"), -1.0
    elif kind == "infinity":
        W.view(-1)[torch.randperm(N * K, generator=g, device=DEV)[:20]] = float("-inf")
    else:
        W *= 1e-36 if kind == "subnormal" else 1e-37
        W.view(-1, 16)[::3, ::2] = 0.0
    Wb = W.to(torch.bfloat16)
    assert kind not in ("nan", "nan blocks", "one nan at the end") or torch.isnan(Wb).any()
    alone = {}
    for f in (dq.FMT_NVFP4, dq.FMT_LUT3, dq.FMT_LUT2):
        alone[f] = [t.clone() for t in dq.export_canonical(dq.pack_weights(Wb, formats=f), f)[:2]]
    for formats in (dq.FMT_NVFP4, dq.FMT_LUT3, dq.FMT_LUT2, dq.FMT_NVFP4 | dq.FMT_LUT3, dq.FMT_NVFP4 | dq.FMT_LUT2, dq.FMT_NVFP4 | dq.FMT_LUT3 | dq.FMT_LUT2):
        for M in (Wb, Wb.float()):
            w = dq.pack_weights(M, formats=formats)
            for f in alone:
                if formats & f:
                    codes, scales, _ = dq.export_canonical(w, f)
                    assert torch.equal(codes, alone[f][0]) and torch.equal(scales, alone[f][1]), (formats, M.dtype, f)
    _status_ok(dq)
