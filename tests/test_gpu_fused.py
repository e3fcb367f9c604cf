"""GPU parity of the fused activation stages (RMSNorm / SiLU(gate)*up in front of the NVFP4 quantiser, App. C.1):
codes and scales bit for bit against the oracle, and the prefill linear built on them against the oracle's fp64
product, through the C ABI."""
import numpy as np
import pytest
import torch

import dq_inputs
from parity_utils import check_outputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def dq():
    import __graft_entry__ as g
    g.build()
    import paper_2609_26333_b200 as dq
    assert torch.cuda.is_available() and torch.cuda.get_device_capability(0) == (10, 0)
    return dq


def _np(t):
    return t.detach().cpu().numpy()


def _status_ok(dq):
    torch.cuda.synchronize()
    st, det = dq.get_status()
    assert st == 0, f"device status {dq.status_string(st)} detail {det}"


def _gamma(K, seed):
    return (dq_inputs.gaussian_bf16(1, K, 0.3, seed)[0].float() + 1.0).to(torch.bfloat16)


@pytest.mark.parametrize("M,K,kind", [(64, 256, "gauss"), (300, 640, "gauss"), (129, 5120, "gauss"), (33, 17408, "student"),
                                        (5, 33024, "gauss")])   # one block per thread, two per thread, the two-pass kernel
def test_rmsnorm_quantiser_bit_exact(dq, oracle, M, K, kind):
    X = dq_inputs.gaussian_bf16(M, K, 1.0, 400 + M) if kind == "gauss" else dq_inputs.student_t_outlier_bf16(M, K, 401)
    X[0] = 0                                              # a zero row: eps keeps it finite
    X[1] = X[1] * 300.0                                   # rows of very different magnitude normalise alike
    gamma = _gamma(K, 402)
    eps = 1e-6
    Xf, gf = dq_inputs.bf16_to_f32_numpy(X), dq_inputs.bf16_to_f32_numpy(gamma[None])[0]
    h = oracle.rmsnorm_bf16(Xf, gf, eps)
    sa = float(np.abs(h).max()) / 2688.0
    big = torch.zeros(M, K + 64, dtype=torch.bfloat16, device=DEV)      # strided rows
    big[:, :K] = X.to(DEV)
    codes, scales = dq.rmsnorm_quantize_activations(big[:, :K], gamma.to(DEV), eps, sa)
    _status_ok(dq)
    rc, rs = oracle.quant_nvfp4(h, sa)
    assert np.array_equal(_np(scales), rs)
    assert np.array_equal(_np(codes), rc)


def test_device_silu_equals_the_cpu_sequence_for_every_bf16_input(dq, oracle):
    """The gate value reaches SiLU as a bf16 number, so there are 65536 inputs: every finite one through the device
    routine (branch-free divide inside its range, the plain divide outside) against the oracle's fp32 sequence, bit for
    bit -- zeros with their sign, denormals, the largest magnitudes."""
    bits = np.arange(65536, dtype=np.uint32)
    finite = ((bits >> 7) & 0xFF) != 0xFF
    bits = bits[finite].astype(np.uint16)
    g = torch.from_numpy(bits.view(np.int16).copy()).view(torch.bfloat16).to(DEV)
    got = dq.test_silu(g).cpu().numpy().view(np.uint32)
    _status_ok(dq)
    gf = (bits.astype(np.uint32) << 16).view(np.float32)
    ref = np.array([oracle.silu_f32(float(x)) for x in gf], dtype=np.float32).view(np.uint32)
    bad = np.flatnonzero(got != ref)
    assert bad.size == 0, f"{bad.size} inputs differ, first g = {gf[bad[0]]!r}: {got[bad[0]]:#x} vs {ref[bad[0]]:#x}"


@pytest.mark.parametrize("M,F", [(64, 256), (300, 640), (130, 17408)])
def test_silu_mul_quantiser_bit_exact(dq, oracle, M, F):
    GU = dq_inputs.gaussian_bf16(M, 2 * F, 2.0, 410 + M)
    GU[0, :16] = 0
    GU[1, :32] = torch.tensor([-200.0, -100.0, -90.0, -88.0, -87.0, -50.0, -20.0, -1e-3, 1e-3, 20.0, 50.0, 87.0, 88.0, 90.0, 100.0, 3e4] * 2)
    h = oracle.silu_mul_bf16(dq_inputs.bf16_to_f32_numpy(GU))
    sa = float(np.abs(h).max()) / 2688.0
    codes, scales = dq.silu_mul_quantize_activations(GU.to(DEV), sa)
    _status_ok(dq)
    rc, rs = oracle.quant_nvfp4(h, sa)
    assert np.array_equal(_np(scales), rs)
    assert np.array_equal(_np(codes), rc)


def test_prefill_linear_on_fused_stages(dq, oracle):
    """RMSNorm -> gate/up projection -> SiLU*up -> down projection, the activation stages fused: each GEMM output
    against the oracle's product of the oracle's quantised operands; same bits as quantising the bf16 intermediate."""
    M, H, F = 320, 512, 1024
    Wgu = dq_inputs.gaussian_bf16(2 * F, H, 0.02, 420)
    Wd = dq_inputs.gaussian_bf16(H, F, 0.02, 421)
    X = dq_inputs.gaussian_bf16(M, H, 1.0, 422)
    gamma = _gamma(H, 423)
    eps = 1e-5
    w_gu = dq.pack_weights(Wgu.to(DEV), formats=dq.FMT_NVFP4)
    w_d = dq.pack_weights(Wd.to(DEV), formats=dq.FMT_NVFP4)
    ref_gu = oracle.pack_weights(dq_inputs.bf16_to_f32_numpy(Wgu))
    ref_d = oracle.pack_weights(dq_inputs.bf16_to_f32_numpy(Wd))
    # stage 1: fused norm + quant, then the gate/up GEMM
    h = oracle.rmsnorm_bf16(dq_inputs.bf16_to_f32_numpy(X), dq_inputs.bf16_to_f32_numpy(gamma[None])[0], eps)
    sa1 = float(np.abs(h).max()) / 2688.0
    ws = dq.alloc_workspace(max(dq.prefill_workspace_bytes(w_gu, M), dq.prefill_workspace_bytes(w_d, M)), DEV)
    GU = torch.empty(M, 2 * F, dtype=torch.bfloat16, device=DEV)
    dq.prefill_rmsnorm_quantize(w_gu, X.to(DEV), gamma.to(DEV), eps, sa1, ws)
    dq.prefill_gemm(w_gu, M, sa1, GU, ws)
    _status_ok(dq)
    Yr, S = oracle.prefill_linear(h, sa1, ref_gu["nvfp4_codes"], ref_gu["nvfp4_scales"], ref_gu["s"])
    check_outputs(GU.float().cpu().numpy().astype(np.float64), Yr, S, "gate/up projection on fused norm + quant")
    # the unfused route gives the same bits
    H_dev = torch.from_numpy(h).to(torch.bfloat16).to(DEV)
    assert torch.equal(dq.prefill_linear(w_gu, H_dev, sa1), GU)
    # stage 2: fused SiLU*up + quant on the GPU's own gate/up output, then the down GEMM
    a2 = oracle.silu_mul_bf16(dq_inputs.bf16_to_f32_numpy(GU.cpu()))
    sa2 = float(np.abs(a2).max()) / 2688.0
    Y = torch.empty(M, H, dtype=torch.bfloat16, device=DEV)
    dq.prefill_silu_mul_quantize(w_d, GU, sa2, ws)
    dq.prefill_gemm(w_d, M, sa2, Y, ws)
    _status_ok(dq)
    Yr, S = oracle.prefill_linear(a2, sa2, ref_d["nvfp4_codes"], ref_d["nvfp4_scales"], ref_d["s"])
    check_outputs(Y.float().cpu().numpy().astype(np.float64), Yr, S, "down projection on fused SiLU*up + quant")
    A2_dev = torch.from_numpy(a2).to(torch.bfloat16).to(DEV)
    assert torch.equal(dq.prefill_linear(w_d, A2_dev, sa2), Y)
    # a row stride below 2 K is rejected before anything is launched
    rc = dq.lib().dq_prefill_silu_mul_quantize(w_d.handle, GU.data_ptr(), M, F, float(sa2), ws.data_ptr(), ws.numel(), None)
    assert rc == 3


def _workspace_codes_scales(ws: torch.Tensor, M: int, F: int):
    """Canonical (rows x F/2 codes, rows x F/16 scales) view of an activation workspace: the codes are stored row-major
    at its start, the scales in 512-byte atoms of 128 rows x 4 blocks (rows r, r+32, r+64, r+96 side by side)."""
    raw = ws.cpu().numpy()
    codes = raw[: M * F // 2].reshape(M, F // 2).copy()
    sf_off = (M * F // 2 + 1023) // 1024 * 1024
    r = np.arange(M)[:, None]
    b = np.arange(F // 16)[None, :]
    off = ((r >> 7) * (F // 64) + (b >> 2)) * 512 + (r & 31) * 16 + ((r & 127) >> 5) * 4 + (b & 3)
    return codes, raw[sf_off + off]


def _e2m1_values(codes: np.ndarray) -> np.ndarray:
    mags = np.array([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0])
    lo, hi = codes & 0xF, codes >> 4
    v = np.empty(codes.shape[:-1] + (codes.shape[-1] * 2,))
    v[..., 0::2] = np.where(lo & 8, -1.0, 1.0) * mags[lo & 7]
    v[..., 1::2] = np.where(hi & 8, -1.0, 1.0) * mags[hi & 7]
    return v


def _e4m3_values(b: np.ndarray) -> np.ndarray:
    e, m = (b >> 3) & 0xF, b & 7
    return np.where(e == 0, m * 2.0 ** -9, (1.0 + m / 8.0) * 2.0 ** (e.astype(np.float64) - 7))


@pytest.mark.parametrize("M,H,F", [(320, 512, 1024), (100, 256, 128), (700, 1024, 2304), (1, 256, 256), (129, 384, 256)])
def test_gate_up_gemm_with_gated_epilogue(dq, oracle, M, H, F):
    """Gate/up GEMM whose epilogue gates and quantises for the down projection (App. C.1): (a) for M > 128 the same bits
    as the GEMM followed by the fused SiLU*up quantiser; (b) against the oracle end to end -- quantised input, fp64
    product, bf16, SiLU*up, NVFP4 -- where the only freedom is the summation order of the GEMM, which moves a bf16
    rounding of G or U now and then and with it, rarely, a code (measured: at most 3 codes in a million, no scale); (c) the down projection on top of it."""
    Wg = dq_inputs.gaussian_bf16(F, H, 0.05, 430)
    Wu = dq_inputs.gaussian_bf16(F, H, 0.05, 431)
    Wd = dq_inputs.gaussian_bf16(H, F, 0.02, 432)
    A = dq_inputs.gaussian_bf16(M, H, 1.0, 433)
    order = dq.gate_up_row_order(F)
    Wgu = torch.cat([Wg, Wu], 0)
    w_il = dq.pack_weights(Wgu[order].contiguous().to(DEV), formats=dq.FMT_NVFP4)       # interleaved rows
    w_d = dq.pack_weights(Wd.to(DEV), formats=dq.FMT_NVFP4)
    sa1 = dq_inputs.static_act_scale(A)
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w_il, M), DEV)
    ows = dq.alloc_workspace(dq.prefill_workspace_bytes(w_d, M), DEV)
    ows.fill_(0xA5)
    dq.prefill_quantize(w_il, A.to(DEV), sa1, ws)
    # the oracle's route: a fused tensor has one global scale, whatever the order of its rows
    ref_gu = oracle.pack_weights(dq_inputs.bf16_to_f32_numpy(Wgu))
    ref_d = oracle.pack_weights(dq_inputs.bf16_to_f32_numpy(Wd))
    Yr, Sr = oracle.prefill_linear(dq_inputs.bf16_to_f32_numpy(A), sa1, ref_gu["nvfp4_codes"], ref_gu["nvfp4_scales"], ref_gu["s"])
    GU_ref = torch.from_numpy(Yr).to(torch.bfloat16)                                     # [gate | up], bf16 as stored
    h_ref = oracle.silu_mul_bf16(dq_inputs.bf16_to_f32_numpy(GU_ref))
    sa2 = float(np.abs(h_ref).max()) / 2688.0
    rc, rs = oracle.quant_nvfp4(h_ref, sa2)
    dq.prefill_gemm_silu_mul_quantize(w_il, M, sa1, ws, w_d, sa2, ows)
    _status_ok(dq)
    codes, scales = _workspace_codes_scales(ows, M, F)
    # (b) against the oracle
    code_diff = np.count_nonzero(((codes ^ rc) & 0x0F) != 0) + np.count_nonzero(((codes ^ rc) & 0xF0) != 0)
    scale_diff = np.count_nonzero(scales != rs)
    assert code_diff <= max(2, 1e-4 * M * F), f"{code_diff} of {M * F} codes differ from the oracle's"
    assert scale_diff <= max(1, 1e-4 * M * F / 16), f"{scale_diff} of {M * F // 16} block scales differ from the oracle's"
    h_gpu = _e2m1_values(codes) * np.repeat(_e4m3_values(scales), 16, axis=1) * sa2
    h_orc = _e2m1_values(rc) * np.repeat(_e4m3_values(rs), 16, axis=1) * sa2
    assert np.linalg.norm(h_gpu - h_orc) <= 1e-3 * np.linalg.norm(h_orc)
    # (a) the two-call path on the same handle: interleaved columns back to [gate | up], then the fused quantiser
    if M > 128:
        GU_il = torch.empty(M, 2 * F, dtype=torch.bfloat16, device=DEV)
        dq.prefill_gemm(w_il, M, sa1, GU_il, ws)
        GU = torch.empty_like(GU_il)
        GU[:, order.to(DEV)] = GU_il
        check_outputs(GU.float().cpu().numpy().astype(np.float64), Yr, Sr, "gate/up, interleaved rows")
        ows2 = dq.alloc_workspace(dq.prefill_workspace_bytes(w_d, M), DEV)
        dq.prefill_silu_mul_quantize(w_d, GU, sa2, ows2)
        _status_ok(dq)
        c2, s2 = _workspace_codes_scales(ows2, M, F)
        assert np.array_equal(codes, c2) and np.array_equal(scales, s2)
    # (c) the down projection reads what the epilogue wrote
    Y = torch.empty(M, H, dtype=torch.bfloat16, device=DEV)
    dq.prefill_gemm(w_d, M, sa2, Y, ows)
    _status_ok(dq)
    Yd, Sd = oracle.prefill_linear(h_ref, sa2, ref_d["nvfp4_codes"], ref_d["nvfp4_scales"], ref_d["s"])
    Yg = Y.float().cpu().numpy().astype(np.float64)
    assert np.linalg.norm(Yg - Yd) <= 2.5e-3 * np.linalg.norm(Yd)          # the bf16 rounding of Y alone is 1.7e-3


def _wide_range(g, rows, K, std):
    """Blocks of 16 whose magnitudes differ by up to 2^9: sums over K that fp32 does not hold exactly, so that their order shows."""
    x = torch.randn(rows, K, generator=g, device=DEV) * std
    e = torch.randint(-9, 1, (rows, K // 16), generator=g, device=DEV)
    return (x * torch.exp2(e.float()).repeat_interleave(16, 1)).to(torch.bfloat16)


@pytest.mark.parametrize("M,H,F", [(300, 17408, 2560), (512, 8192, 256), (1000, 17408, 2560), (300, 4096, 128), (129, 5120, 512),
                                   (257, 2048, 128), (129, 4096, 512), (129, 8192, 896), (129, 8192, 1280), (129, 8192, 1408),
                                   (129, 8192, 1664), (200, 8192, 1920), (257, 8192, 1664), (2048, 5120, 2560)])
def test_gated_epilogue_adds_up_as_the_plain_gemm_does(dq, M, H, F):
    """The same bits as the two calls also where the GEMM shares a tile's k-steps out over a cluster or splits its columns over two
    launches, on operands whose sums depend on the order they are taken in."""
    g = torch.Generator(device=DEV).manual_seed(M + H)
    w_gu = dq.pack_weights(_wide_range(g, 2 * F, H, 0.02), formats=dq.FMT_NVFP4)
    w_d = dq.pack_weights((torch.randn(128, F, generator=g, device=DEV) * 0.02).to(torch.bfloat16), formats=dq.FMT_NVFP4)
    A = _wide_range(g, M, H, 1.0)
    sa = float(A.abs().max()) / 2688.0
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w_gu, M), DEV)
    out, want = (dq.alloc_workspace(dq.prefill_workspace_bytes(w_d, M), DEV) for _ in range(2))
    dq.prefill_quantize(w_gu, A, sa, ws)
    Y = torch.empty(M, 2 * F, dtype=torch.bfloat16, device=DEV)
    dq.prefill_gemm(w_gu, M, sa, Y, ws)
    GU = torch.empty_like(Y)
    GU[:, dq.gate_up_row_order(F).to(DEV)] = Y
    s_out = float((torch.nn.functional.silu(GU[:, :F].float()) * GU[:, F:].float()).abs().max()) / 2688.0
    out.fill_(0xA5)
    want.fill_(0xA5)
    dq.prefill_silu_mul_quantize(w_d, GU, s_out, want)
    dq.prefill_gemm_silu_mul_quantize(w_gu, M, sa, ws, w_d, s_out, out)
    _status_ok(dq)
    assert torch.equal(out, want)


def test_gate_up_gemm_with_gated_epilogue_arguments(dq):
    F, H, M = 256, 256, 64
    w_gu = dq.pack_weights(dq_inputs.gaussian_bf16(2 * F, H, 0.05, 440).to(DEV), formats=dq.FMT_NVFP4)
    w_d = dq.pack_weights(dq_inputs.gaussian_bf16(H, F, 0.02, 441).to(DEV), formats=dq.FMT_NVFP4)
    w_bad = dq.pack_weights(dq_inputs.gaussian_bf16(H, 2 * F, 0.02, 442).to(DEV), formats=dq.FMT_NVFP4)
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w_gu, M), DEV)
    ows = dq.alloc_workspace(dq.prefill_workspace_bytes(w_bad, M), DEV)
    call = dq.lib().dq_prefill_gemm_silu_mul_quantize
    assert call(w_gu.handle, M, 1.0, ws.data_ptr(), ws.numel(), w_bad.handle, 1.0, ows.data_ptr(), ows.numel(), None) == 2   # shape
    assert call(w_gu.handle, M, 1.0, ws.data_ptr(), ws.numel(), w_d.handle, 0.0, ows.data_ptr(), ows.numel(), None) == 1     # scale
    assert call(w_gu.handle, M, 1.0, ws.data_ptr(), ws.numel(), w_d.handle, 1.0, ows.data_ptr(), 1024, None) == 4            # workspace
    assert call(w_gu.handle, M, 1.0, ws.data_ptr(), ws.numel(), w_d.handle, 1.0, ws.data_ptr(), ws.numel(), None) == 1       # overlap
    assert call(w_gu.handle, M, 1.0, ws.data_ptr(), ws.numel(), None, 1.0, ows.data_ptr(), ows.numel(), None) == 1
    _status_ok(dq)


def test_gated_ffn_on_lut3_only_handles_and_from_a_cuda_graph(dq):
    """The gated chain on handles that store LUT3 only (both projections cast to NVFP4 per call, Sec. 2.3) gives, bit
    for bit, what handles with the pack-time NVFP4 view give; captured in a CUDA graph and replayed on new activations
    it gives what the eager calls give."""
    M, H, F = 384, 512, 768
    order = dq.gate_up_row_order(F)
    Wgu = torch.cat([dq_inputs.gaussian_bf16(F, H, 0.05, 450), dq_inputs.gaussian_bf16(F, H, 0.05, 451)], 0)[order].contiguous().to(DEV)
    Wd = dq_inputs.gaussian_bf16(H, F, 0.02, 452).to(DEV)
    A = dq_inputs.gaussian_bf16(M, H, 1.0, 453).to(DEV)
    sa1, sa2 = 5.0 / 2688.0, 2.0 / 2688.0
    outs = []
    for fmt in (dq.FMT_LUT3, dq.FMT_NVFP4_FROM_LUT3):
        w_gu, w_d = dq.pack_weights(Wgu, formats=fmt), dq.pack_weights(Wd, formats=fmt)
        ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w_gu, M), DEV)
        ows = dq.alloc_workspace(dq.prefill_workspace_bytes(w_d, M), DEV)
        ws.fill_(0xFF); ows.fill_(0xFF)
        Y = torch.empty(M, H, dtype=torch.bfloat16, device=DEV)

        def chain():
            dq.prefill_quantize(w_gu, A, sa1, ws)
            dq.prefill_gemm_silu_mul_quantize(w_gu, M, sa1, ws, w_d, sa2, ows)
            dq.prefill_gemm(w_d, M, sa2, Y, ows)

        chain()
        _status_ok(dq)
        outs.append(Y.clone())
        if fmt == dq.FMT_LUT3:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                chain()
            A0 = A.clone()
            A.copy_(dq_inputs.gaussian_bf16(M, H, 1.0, 454).to(DEV))
            Y.zero_()
            graph.replay()
            torch.cuda.synchronize()
            got = Y.clone()
            chain()
            _status_ok(dq)
            assert torch.equal(got, Y)
            assert not torch.equal(got, outs[0])
            A.copy_(A0)
    assert torch.equal(outs[0], outs[1])
    assert float(outs[0].float().abs().max()) > 0.0
