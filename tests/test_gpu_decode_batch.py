"""GPU parity of the batch decode kernel (dequantised weights through tensor memory) against the CPU oracle, with the
tolerances of parity_utils: every encoding, every column padding, ragged rows and row lengths, one and several CTAs a tile."""
import numpy as np
import pytest
import torch

import dq_inputs
from parity_utils import check_outputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TC = 5                                   # test-hook variant: this kernel whatever the batch


@pytest.fixture(scope="module")
def dq():
    import __graft_entry__ as g
    g.build()
    import paper_2609_26333_b200 as dq
    return dq


def _status_ok(dq):
    torch.cuda.synchronize()
    st, det = dq.get_status()
    assert st == 0, f"device status {dq.status_string(st)} detail {det}"


_cache = {}


def _layer(oracle, N, K):
    if (N, K) not in _cache:
        W = dq_inputs.gaussian_bf16(N, K, 0.02, 500 + N + K)
        Wf = dq_inputs.bf16_to_f32_numpy(W)
        ref = oracle.pack_weights(Wf)
        ref["lut2_planes"], ref["lut2_scales"] = oracle.quant_lut2(Wf, ref["s"])
        _cache[(N, K)] = (W, ref)
    return _cache[(N, K)]


def _reference(oracle, ref, fmt, X):
    Xf = dq_inputs.bf16_to_f32_numpy(X)
    if fmt == "lut3":
        return oracle.decode_linear(Xf, ref["lut3_planes"], ref["lut3_scales"], ref["s"])
    if fmt == "lut2":
        return oracle.decode_linear_lut2(Xf, ref["lut2_planes"], ref["lut2_scales"], ref["s"])
    return oracle.decode_linear_nvfp4(Xf, ref["nvfp4_codes"], ref["nvfp4_scales"], ref["s"])


def _f64(t):
    return t.detach().float().cpu().numpy().astype(np.float64)


# one row tile and less, the last half tile missing or ragged, K inside a slice of 512 and inside a 128-weight pair
SHAPES = [(16, 128), (144, 384), (272, 640), (400, 1152), (1040, 2048)]


@pytest.mark.parametrize("fmt", ["lut3", "lut2", "nvfp4"])
@pytest.mark.parametrize("N,K", SHAPES)
@pytest.mark.parametrize("B", [1, 9, 16, 17, 33, 48, 64])
def test_decode_batch_parity(dq, oracle, fmt, N, K, B):
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 900 + B)
    Yr, S = _reference(oracle, ref, fmt, X)
    big = torch.zeros(B, K + 24, dtype=torch.bfloat16, device=DEV)        # strided activations, guarded strided outputs
    big[:, :K] = X.to(DEV)
    out = torch.full((B + 1, N + 8), 7.0, dtype=torch.bfloat16, device=DEV)
    dq.test_decode_linear(w, code, big[:, :K], out=out[:B, :N], variant=TC)
    _status_ok(dq)
    check_outputs(_f64(out[:B, :N]), Yr, S, f"{fmt} {B}x{N}x{K}")
    assert torch.all(out[B] == 7.0) and torch.all(out[:, N:] == 7.0)
    if B > 8:                                                             # what the public entry point runs
        y = {"lut3": dq.decode_linear, "lut2": dq.decode_linear_lut2, "nvfp4": dq.decode_linear_nvfp4}[fmt](w, X.to(DEV))
        _status_ok(dq)
        check_outputs(_f64(y), Yr, S, f"{fmt} {B}x{N}x{K} public")


@pytest.mark.parametrize("fmt", ["lut3", "nvfp4"])
@pytest.mark.parametrize("csize", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("B", [10, 40, 61])
def test_decode_batch_ctas_per_tile(dq, oracle, fmt, csize, B):
    N, K = 784, 4224                                                      # nine slices, the last one short
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "nvfp4": dq.FMT_NVFP4}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 700 + B)
    Yr, S = _reference(oracle, ref, fmt, X)
    outs = []
    for _ in range(2):
        y = torch.full((B, N), float("nan"), dtype=torch.bfloat16, device=DEV)
        dq.test_decode_linear(w, code, X.to(DEV), out=y, variant=TC, warps_per_group=csize)
        outs.append(y)
    _status_ok(dq)
    check_outputs(_f64(outs[0]), Yr, S, f"{fmt} {csize} CTAs a tile, batch {B}")
    assert torch.equal(outs[0], outs[1])                                  # sums in a fixed order


@pytest.mark.parametrize("fmt", ["lut3", "lut2", "nvfp4"])
def test_decode_batch_wide_range_and_sparse_activations(dq, oracle, fmt):
    """Columns that differ by 2^60, elements down to 2^-28 of a slice's largest, zero columns, single non-zeros."""
    N, K, B = 272, 1152, 20
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 77).float()
    g = torch.Generator().manual_seed(5)
    X *= torch.pow(2.0, torch.randint(-20, 1, (B, K), generator=g).float())
    X *= torch.pow(2.0, torch.linspace(-30, 30, B).round())[:, None]
    X[3] = 0
    X[4, 1:] = 0
    X[5, :1000] = 0
    X = X.to(torch.bfloat16)
    Yr, S = _reference(oracle, ref, fmt, X)
    y = dq.test_decode_linear(w, code, X.to(DEV), variant=TC)
    _status_ok(dq)
    Y = _f64(y)
    for b in range(B):                                                    # per column: the Frobenius check must not hide small ones
        check_outputs(Y[b:b + 1], Yr[b:b + 1], S[b:b + 1], f"{fmt} column {b}")
    # one-hot columns: the weight itself, rounded to bf16 once
    E = torch.zeros(16, K, dtype=torch.bfloat16)
    ks = [0, 3, 4, 15, 16, 37, 127, 128, 511, 512, 639, 640, 1000, 1023, 1024, 1151]
    E[torch.arange(16), torch.tensor(ks)] = 1.0
    Yr, _ = _reference(oracle, ref, fmt, E)
    y = dq.test_decode_linear(w, code, E.to(DEV), variant=TC)
    _status_ok(dq)
    assert torch.equal(y.float().cpu(), torch.from_numpy(Yr).to(torch.float32).to(torch.bfloat16).float())


def test_decode_batch_fine_codebook_takes_the_general_path(dq, oracle):
    """Levels that are not multiples of 2^-15 do not fit the kernel's pair of fp16 numbers under every block scale."""
    N, K, B = 272, 640, 12
    W, _ = _layer(oracle, N, K)
    cb = torch.tensor([-4.0, -2.0, -0.001, 0.0, 0.0011, 2.5, 4.0, 6.0], dtype=torch.float16)
    bits = [int(v) & 0xFFFF for v in cb.view(torch.int16)]
    w = dq.pack_weights(W.to(DEV), formats=dq.FMT_LUT3, codebook_f16=bits)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 12).to(DEV)
    with pytest.raises(dq.DQError):
        dq.test_decode_linear(w, dq.FMT_LUT3, X, variant=TC)
    planes, scales, s = dq.export_canonical(w, dq.FMT_LUT3)
    bit = (planes.long()[:, :, :, None] >> torch.arange(32, device=DEV)) & 1
    idx = (bit[:, 0] + 2 * bit[:, 1] + 4 * bit[:, 2]).flatten(1)
    Wd = cb.double().to(DEV)[idx] * scales.view(torch.float8_e4m3fn).double().repeat_interleave(16, dim=1) * s.double()
    Y = dq.decode_linear(w, X)
    _status_ok(dq)
    check_outputs(_f64(Y), (X.double() @ Wd.T).cpu().numpy(), (X.double().abs() @ Wd.abs().T).cpu().numpy(), "fine codebook")


def _imported_layer(dq, N, K, cb, seed):
    """A LUT3 handle from random indices and every finite block scale, as an import may bring them, and its weights in fp64."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    planes = torch.randint(-2 ** 31, 2 ** 31, (N, 3, K // 32), generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
    scales = torch.randint(0, 256, (N, K // 16), generator=g, device=DEV, dtype=torch.int32)
    scales = (scales - ((scales & 0x7F) == 0x7F).int()).to(torch.uint8)                # 0x7F and 0xFF are NaN
    scales[:, :2] = 0x7E                                                               # the largest, 448
    s = 2.0 ** -10
    w = dq.import_canonical(N, K, dq.FMT_LUT3, s, lut3=(planes, scales), codebook_f16=[int(v) & 0xFFFF for v in cb.view(torch.int16)])
    bit = (planes.long()[:, :, :, None] >> torch.arange(32, device=DEV)) & 1
    idx = (bit[:, 0] + 2 * bit[:, 1] + 4 * bit[:, 2]).flatten(1)
    return w, cb.double().to(DEV)[idx] * scales.view(torch.float8_e4m3fn).double().repeat_interleave(16, dim=1) * s


@pytest.mark.parametrize("lowest,fits", [(-146.0, True), (-146.25, False), (-200.0, False), (-65504.0, False)])
@pytest.mark.parametrize("N,K", [(512, 256), (512, 1024), (272, 640)])
@pytest.mark.parametrize("B", [5, 9, 40])
def test_decode_batch_codebooks_of_large_magnitude(dq, lowest, fits, N, K, B):
    """The negative side of a codebook has no limit.  A level times the largest block scale, 448, fits fp16 up to 146.2; beyond, the
    kernel refuses and the public call takes one that multiplies in fp32."""
    w, Wd = _imported_layer(dq, N, K, torch.tensor([lowest, -2.0, -1.0, 0.0, 1.0, 2.5, 4.0, 6.0], dtype=torch.float16), 31 + N + K)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 40 + B).to(DEV)
    Yr, S = (X.double() @ Wd.T).cpu().numpy(), (X.double().abs() @ Wd.abs().T).cpu().numpy()
    Y = dq.decode_linear(w, X)
    _status_ok(dq)
    check_outputs(_f64(Y), Yr, S, f"lowest level {lowest}, batch {B}")
    if fits:
        Y = dq.test_decode_linear(w, dq.FMT_LUT3, X, variant=TC)
        _status_ok(dq)
        check_outputs(_f64(Y), Yr, S, f"lowest level {lowest}, batch {B}, batch kernel")
    else:
        with pytest.raises(dq.DQError):
            dq.test_decode_linear(w, dq.FMT_LUT3, X, variant=TC)


def _dequantised(dq, w, fmt):
    """The handle's weights in fp64 on the GPU, from its canonical export."""
    codes, scales, s = dq.export_canonical(w, {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt])
    if fmt == "nvfp4":
        mags = torch.tensor([0, 0.5, 1, 1.5, 2, 3, 4, 6], dtype=torch.float64, device=DEV)
        levels = torch.cat([mags, -mags])
        idx = torch.stack([codes & 15, codes >> 4], dim=2).flatten(1).long()
    else:
        lo = {"lut3": [-4.703125, -2.869140625, -1.369140625, 0, 1.220703125, 2.529296875, 4.046875, 6],
              "lut2": [-3.65234375, 0, 2.5234375, 6]}[fmt]
        levels = torch.tensor(lo, dtype=torch.float64, device=DEV)
        bit = (codes[:, :, :, None] >> torch.arange(32, device=DEV, dtype=torch.int32)) & 1
        idx = sum(bit[:, p].int() << p for p in range(codes.shape[1])).flatten(1).long()
    return levels[idx] * scales.view(torch.float8_e4m3fn).double().repeat_interleave(16, dim=1) * s.double()


@pytest.mark.parametrize("fmt", ["lut3", "lut2", "nvfp4"])
@pytest.mark.parametrize("B", [9, 40])
@pytest.mark.parametrize("rest", [16, 128, 144])
def test_decode_batch_last_tile_of_a_cta_has_one_half(dq, fmt, B, rest):
    """More 256-row tiles than SMs and a last one with rows in its first half only (and, beside it, in both): a CTA then takes a
    full tile and a half one, the second half's warps reading the full one back while the half one is under way.  Slices whose
    magnitudes differ by many binades: an inverse scale of another slice would show."""
    N, K = 256 * torch.cuda.get_device_properties(0).multi_processor_count + rest, 2688
    g = torch.Generator(device=DEV).manual_seed(N + B)
    W = (torch.randn(N, K, generator=g, device=DEV) * 0.02).to(torch.bfloat16)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt]
    w = dq.pack_weights(W, formats=code)
    X = torch.randn(B, K, generator=g, device=DEV) * torch.exp2(3.0 * torch.arange(K, device=DEV).div(512, rounding_mode="floor"))
    X = X.to(torch.bfloat16)
    Wd = _dequantised(dq, w, fmt)
    Yr, S = (X.double() @ Wd.T).cpu().numpy(), (X.double().abs() @ Wd.abs().T).cpu().numpy()
    for _ in range(3):
        y = dq.test_decode_linear(w, code, X, variant=TC)
        _status_ok(dq)
        check_outputs(_f64(y), Yr, S, f"{fmt} {B}x{N}x{K}")


@pytest.mark.parametrize("fmt", ["lut3", "lut2", "nvfp4"])
@pytest.mark.parametrize("B", [9, 40])
def test_decode_batch_infinite_and_huge_activations(dq, fmt, B):
    """An infinite activation gives what its products give: an infinity where the weight is not zero, NaN where it is, as with one
    column; infinities of several 128-weight groups add up; the columns beside it are not touched.  NaN stays in its column.
    Huge finite magnitudes are scaled like any other."""
    N, K = 272, 1152
    g = torch.Generator(device=DEV).manual_seed(61 + B)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt]
    w = dq.pack_weights((torch.randn(N, K, generator=g, device=DEV) * 0.02).to(torch.bfloat16), formats=code)
    call = {"lut3": dq.decode_linear, "lut2": dq.decode_linear_lut2, "nvfp4": dq.decode_linear_nvfp4}[fmt]
    Wd = _dequantised(dq, w, fmt)
    X = torch.randn(B, K, generator=g, device=DEV).to(torch.bfloat16)
    Y0 = dq.test_decode_linear(w, code, X, variant=TC)
    X[0, 700] = float("inf")
    X[1, 3] = float("-inf")
    X[2, 129], X[2, 1151] = float("inf"), float("-inf")
    X[3, 64] = float("nan")
    X[4] *= 2.0 ** 104                                        # the sums, before the tensor scale of about 2^-15, stay below 2^128
    X[5] = 0
    X[5, 17] = 2.0 ** 115
    Y = dq.test_decode_linear(w, code, X, variant=TC)
    _status_ok(dq)
    Yr = X.double() @ Wd.T                                    # 0 times infinity is NaN there too
    for b in range(3):
        assert not torch.isfinite(Yr[b]).any()
        assert torch.equal(torch.isnan(Y[b]), torch.isnan(Yr[b])), f"column {b}"
        assert torch.equal(Y[b].double().nan_to_num(0.0, 1.0, -1.0), Yr[b].nan_to_num(0.0, 1.0, -1.0)), f"column {b}"
    assert torch.isnan(Y[3]).all()
    S = X.double().abs() @ Wd.abs().T
    for b in (4, 5):
        check_outputs(_f64(Y[b:b + 1]), Yr[b:b + 1].cpu().numpy(), S[b:b + 1].cpu().numpy(), f"column {b}")
    assert torch.equal(Y[6:], Y0[6:])
    one = call(w, X[:1])
    _status_ok(dq)
    assert torch.equal(torch.isnan(one[0]), torch.isnan(Y[0])) and torch.equal(one[0].nan_to_num(0.0), Y[0].nan_to_num(0.0))


def test_decode_batch_wait_runs_out(dq):
    """A ring stage that is never requested: the waits run out, the launch returns and reports."""
    w = dq.pack_weights(dq_inputs.gaussian_bf16(256, 512, 0.02, 1).to(DEV), formats=dq.FMT_LUT3)
    X = dq_inputs.gaussian_bf16(12, 512, 1.0, 2).to(DEV)
    good = dq.decode_linear(w, X)
    dq.test_decode_linear(w, dq.FMT_LUT3, X, variant=1, wait_cycles=2_000_000)
    torch.cuda.synchronize()
    st, _ = dq.get_status()
    assert dq.status_string(st) == "device-side wait ran out"
    assert torch.equal(dq.decode_linear(w, X), good)
    _status_ok(dq)


@pytest.mark.parametrize("N,K,B", [(1024, 1024, 4), (1024, 1024, 6), (1024, 1024, 12), (8192, 2048, 12), (2048, 2048, 24), (4096, 512, 40)])
def test_decode_left_out_copy_is_missed_at_every_batch(dq, N, K, B):
    """The hook that leaves a copy out does so whichever kernel the shape would take."""
    w = dq.pack_weights(dq_inputs.gaussian_bf16(N, K, 0.02, 1).to(DEV), formats=dq.FMT_LUT3)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 2).to(DEV)
    good = dq.decode_linear(w, X)
    dq.test_decode_linear(w, dq.FMT_LUT3, X, variant=1, wait_cycles=2_000_000)
    torch.cuda.synchronize()
    st, _ = dq.get_status()
    assert dq.status_string(st) == "device-side wait ran out"
    assert torch.equal(dq.decode_linear(w, X), good)
    _status_ok(dq)


@pytest.mark.parametrize("fmt", ["lut3", "lut2"])
@pytest.mark.parametrize("N,K", SHAPES + [(4112, 1536)])
@pytest.mark.parametrize("B", [1, 5, 8])
def test_decode_rows16_parity(dq, oracle, fmt, N, K, B):
    """The kernel with 16-row tiles (what batches of five to eight take): ragged slices, one and several warps per tile, more tiles
    than one round takes."""
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 300 + B)
    Yr, S = _reference(oracle, ref, fmt, X)
    out = torch.full((B + 1, N + 8), 7.0, dtype=torch.bfloat16, device=DEV)
    dq.test_decode_linear(w, code, X.to(DEV), out=out[:B, :N], variant=6)
    _status_ok(dq)
    check_outputs(_f64(out[:B, :N]), Yr, S, f"{fmt} {B}x{N}x{K}")
    assert torch.all(out[B] == 7.0) and torch.all(out[:, N:] == 7.0)
    if B > 4:
        y = {"lut3": dq.decode_linear, "lut2": dq.decode_linear_lut2}[fmt](w, X.to(DEV))
        _status_ok(dq)
        check_outputs(_f64(y), Yr, S, f"{fmt} {B}x{N}x{K} public")


@pytest.mark.parametrize("fmt,N,K,B,rows16", [("lut3", 19216, 640, 7, True), ("lut2", 10304, 1664, 8, True), ("lut3", 4464, 4608, 5, True),
                                              ("lut2", 464, 6144, 6, None), ("lut2", 496, 7552, 5, False)])
def test_decode_line_between_row_tiles(dq, oracle, fmt, N, K, B, rows16):
    """Both sides of the line between 8-row and 16-row tiles: the public call against the oracle, and bit for bit the 16-row kernel where
    that is the one taken."""
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 700 + B)
    Yr, S = _reference(oracle, ref, fmt, X)
    y = {"lut3": dq.decode_linear, "lut2": dq.decode_linear_lut2}[fmt](w, X.to(DEV))
    forced = dq.test_decode_linear(w, code, X.to(DEV), variant=6)
    _status_ok(dq)
    check_outputs(_f64(y), Yr, S, f"{fmt} {B}x{N}x{K} public")
    check_outputs(_f64(forced), Yr, S, f"{fmt} {B}x{N}x{K} 16 rows")
    if rows16:
        assert torch.equal(y, forced)


@pytest.mark.parametrize("fmt", ["lut3", "lut2", "nvfp4"])
@pytest.mark.parametrize("N,K", [(512, 256), (528, 1024), (1024, 2176), (2384, 640)])
@pytest.mark.parametrize("B", [4, 6, 9, 16, 24])
def test_decode_takes_any_kernel_on_few_rows(dq, oracle, fmt, N, K, B):
    """Small matrices on both sides of the lines between the kernels, through the public calls."""
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt]
    call = {"lut3": dq.decode_linear, "lut2": dq.decode_linear_lut2, "nvfp4": dq.decode_linear_nvfp4}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 700 + B)
    Yr, S = _reference(oracle, ref, fmt, X)
    out = torch.full((B + 1, N + 8), 7.0, dtype=torch.bfloat16, device=DEV)
    call(w, X.to(DEV), out=out[:B, :N])
    _status_ok(dq)
    check_outputs(_f64(out[:B, :N]), Yr, S, f"{fmt} {B}x{N}x{K}")
    assert torch.all(out[B] == 7.0) and torch.all(out[:, N:] == 7.0)


@pytest.mark.parametrize("fmt", ["lut3", "lut2"])
@pytest.mark.parametrize("N,K", [(1040, 1024), (528, 2048), (2064, 640)])
@pytest.mark.parametrize("B", [9, 16, 24, 29])
def test_decode_columns_of_very_different_magnitude(dq, oracle, fmt, N, K, B):
    """Columns that differ by 2^60 in the slice-by-slice kernel, whatever shares its pass, and through the public call, where these
    shapes reach it."""
    W, ref = _layer(oracle, N, K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2}[fmt]
    w = dq.pack_weights(W.to(DEV), formats=code)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 800 + B).float()
    X = (X * torch.pow(2.0, torch.linspace(-30, 30, B).round())[:, None]).to(torch.bfloat16)
    X[3] = 0
    X[4, 300:] = 0
    Yr, S = _reference(oracle, ref, fmt, X)
    call = {"lut3": dq.decode_linear, "lut2": dq.decode_linear_lut2}[fmt]
    for Y in (_f64(dq.test_decode_linear(w, code, X.to(DEV), variant=4)), _f64(call(w, X.to(DEV)))):
        _status_ok(dq)
        for b in range(B):
            check_outputs(Y[b:b + 1], Yr[b:b + 1], S[b:b + 1], f"{fmt} {B}x{N}x{K} column {b}")


def test_decode_nvfp4_hook_refuses_what_it_does_not_know(dq):
    """Variants that do not exist for this encoding and cluster sizes that do not fit are argument errors, not another kernel's run."""
    N, K = 272, 1024
    w = dq.pack_weights(dq_inputs.gaussian_bf16(N, K, 0.02, 3).to(DEV), formats=dq.FMT_NVFP4)
    X = dq_inputs.gaussian_bf16(2, K, 1.0, 4).to(DEV)
    for kw in ({"variant": -1}, {"variant": 2}, {"variant": 3}, {"variant": 4}, {"variant": 7}, {"variant": 99},
               {"variant": TC, "warps_per_group": 3}, {"variant": TC, "warps_per_group": 9}, {"variant": TC, "warps_per_group": -1}):
        with pytest.raises(dq.DQError) as e:
            dq.test_decode_linear(w, dq.FMT_NVFP4, X, **kw)
        assert e.value.code == 1, kw
    for variant in (0, 1, TC, 6):
        dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=variant)
    _status_ok(dq)


@pytest.mark.parametrize("N,K", [(16, 128), (144, 384), (784, 1152), (272, 7168), (400, 9216), (144, 17408), (48, 21632), (80, 32768)])
@pytest.mark.parametrize("B", [1, 3, 8, 17])
def test_decode_nvfp4_every_kernel(dq, oracle, N, K, B):
    """The NVFP4 kernels at every ring depth of the mma.sync kernel (one warp a row group up to 32), in one pass over the columns and in
    several, whichever of them the public call would take."""
    W, ref = _layer(oracle, N, K)
    w = dq.pack_weights(W.to(DEV), formats=dq.FMT_NVFP4)
    X = dq_inputs.gaussian_bf16(B, K, 1.0, 950 + B)
    Yr, S = _reference(oracle, ref, "nvfp4", X)
    for variant in (0, 1, TC, 6):
        out = torch.full((B + 1, N + 8), 7.0, dtype=torch.bfloat16, device=DEV)
        dq.test_decode_linear(w, dq.FMT_NVFP4, X.to(DEV), out=out[:B, :N], variant=variant)
        _status_ok(dq)
        check_outputs(_f64(out[:B, :N]), Yr, S, f"variant {variant}, {B}x{N}x{K}")
        assert torch.all(out[B] == 7.0) and torch.all(out[:, N:] == 7.0)


def _decode_calls(dq, w, X):
    """Calls that reach the batch kernel, the 16-row kernel and the slice-by-slice kernel, and what the public entry points take."""
    calls = [(dq.FMT_LUT3, X[:9], TC), (dq.FMT_LUT3, X[:7], 6), (dq.FMT_LUT3, X[:20], 4), (dq.FMT_LUT2, X[:24], TC), (dq.FMT_LUT2, X[:5], 6),
             (dq.FMT_LUT2, X[:33], 4), (dq.FMT_NVFP4, X[:6], TC), (dq.FMT_NVFP4, X[:2], 6)]
    calls += [(f, X[:b], 0) for f in (dq.FMT_LUT3, dq.FMT_LUT2, dq.FMT_NVFP4) for b in (6, 12, 40)]
    return [lambda out, f=f, x=x, v=v, **kw: dq.test_decode_linear(w, f, x, out=out, variant=v, **kw) for f, x, v in calls], \
        [x.shape[0] for _, x, _ in calls]


@pytest.mark.parametrize("N,K", [(1040, 2048), (144, 4224)])
def test_decode_kernels_replay_from_a_cuda_graph(dq, N, K):
    """Every decode kernel captured in one graph, launch after launch; replays on new activations give what eager calls give."""
    w = dq.pack_weights(dq_inputs.gaussian_bf16(N, K, 0.02, 11).to(DEV), formats=dq.FMT_NVFP4 | dq.FMT_LUT3 | dq.FMT_LUT2)
    X = dq_inputs.gaussian_bf16(40, K, 1.0, 12).to(DEV)
    calls, rows = _decode_calls(dq, w, X)
    outs = [torch.zeros(b, N, dtype=torch.bfloat16, device=DEV) for b in rows]
    for call, y in zip(calls, outs):
        call(y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for call, y in zip(calls, outs):
            call(y)
    for seed in (13, 14):
        X.copy_(dq_inputs.gaussian_bf16(40, K, 1.0, seed).to(DEV))
        for y in outs:
            y.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for call, y in zip(calls, outs):
            got = y.clone()
            call(y)
            torch.cuda.synchronize()
            assert torch.equal(got, y) and float(got.float().abs().max()) > 0.0
    _status_ok(dq)


def test_decode_kernels_on_several_streams_at_once(dq):
    """Every decode kernel on three streams at a time, on one handle: the bits of the calls one after the other."""
    N, K = 1040, 2048
    w = dq.pack_weights(dq_inputs.gaussian_bf16(N, K, 0.02, 15).to(DEV), formats=dq.FMT_NVFP4 | dq.FMT_LUT3 | dq.FMT_LUT2)
    streams = [torch.cuda.Stream(device=DEV) for _ in range(3)]
    work, want = [], []
    for i in range(3):
        calls, rows = _decode_calls(dq, w, dq_inputs.gaussian_bf16(40, K, 1.0, 16 + i).to(DEV))
        work.append((calls, [torch.zeros(b, N, dtype=torch.bfloat16, device=DEV) for b in rows]))
        want.append([call(torch.empty(b, N, dtype=torch.bfloat16, device=DEV)) for call, b in zip(calls, rows)])
    torch.cuda.synchronize()
    for _ in range(4):
        for i, st in enumerate(streams):
            with torch.cuda.stream(st):
                for call, y in zip(*work[i]):
                    call(y, stream=st)
    torch.cuda.synchronize()
    _status_ok(dq)
    for i in range(3):
        for y, z in zip(work[i][1], want[i]):
            assert torch.equal(y, z)


@pytest.mark.parametrize("fmt,limit", [("lut3", 6e-4), ("lut2", 6e-4), ("nvfp4", 3e-4)])
@pytest.mark.parametrize("K", [512, 2048, 5120, 17408])
def test_decode_batch_share_of_misrounded_outputs(dq, fmt, limit, K):
    """Outputs that differ from the exact sum rounded to bf16 once.  A sum that is off by e ulp of fp32 moves a rounding with probability
    e * 2^-15 (half a bf16 step is 2^15 fp32 ulp of a sum without cancellation, fewer with it): measured 1.6e-4 to 2.8e-4 for the LUT formats in groups
    of 128 weights and 0.4e-4 to 1.2e-4 for NVFP4; the mma.sync kernels 0.9e-4 to 3.1e-4 and 0.6e-4 to 1.6e-4.  Groups of 512
    gave the LUT formats 7e-4.  The limits are at least twice the largest; 655360 outputs scatter by about 0.2e-4."""
    N, B = 10240, 64
    g = torch.Generator(device=DEV).manual_seed(K)
    code = {"lut3": dq.FMT_LUT3, "lut2": dq.FMT_LUT2, "nvfp4": dq.FMT_NVFP4}[fmt]
    w = dq.pack_weights((torch.randn(N, K, generator=g, device=DEV) * 0.02).to(torch.bfloat16), formats=code)
    X = torch.randn(B, K, generator=g, device=DEV).to(torch.bfloat16)
    y = dq.test_decode_linear(w, code, X, variant=TC)
    _status_ok(dq)
    exact = (X.double() @ _dequantised(dq, w, fmt).T).to(torch.float32).to(torch.bfloat16)
    share = float((y != exact).double().mean())
    assert share < limit, f"{share:.2e}"
