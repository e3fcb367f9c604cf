"""NVFP4 decode through the FP4 tensor cores: activations as digits, with and without a workspace, against the dequantised matrix in
double precision, at ragged sizes, every cluster size and magnitudes where digits can go wrong."""
import numpy as np
import pytest
import torch

from parity_utils import check_outputs
from test_gpu_decode_batch import DEV, _dequantised, _f64, _status_ok, dq  # noqa: F401

pytestmark = pytest.mark.gpu
FP4 = 8


def _pack(dq, N, K, seed):  # noqa: F811
    g = torch.Generator(device=DEV).manual_seed(seed)
    w = dq.pack_weights((torch.randn(N, K, generator=g, device=DEV) * 0.02).to(torch.bfloat16), formats=dq.FMT_NVFP4)
    return g, w, _dequantised(dq, w, "nvfp4")


def _call(dq, w, X, csize=0):  # noqa: F811
    if X.shape[0] <= 4:
        return dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=FP4, warps_per_group=csize)
    ws = torch.full((dq.decode_nvfp4_workspace_bytes(w, X.shape[0], True) + 512,), 255, dtype=torch.uint8, device=DEV)
    n = ws.numel() - 512
    Y = dq.decode_linear_nvfp4_ws(w, X, ws[:n])
    assert (ws[n:] == 255).all()
    return Y


def _check(Y, X, Wd, what):
    check_outputs(_f64(Y), (X.double() @ Wd.T).cpu().numpy(), (X.double().abs() @ Wd.abs().T).cpu().numpy(), what)


@pytest.mark.parametrize("B", [1, 3, 4, 5, 8, 9, 13, 16])
@pytest.mark.parametrize("N,K", [(16, 128), (256, 256), (272, 384), (1040, 1152), (512, 2176), (240, 8320), (40000, 256)])
def test_fp4_decode_ragged_sizes(dq, N, K, B):  # noqa: F811
    g, w, Wd = _pack(dq, N, K, N + K)
    wide = torch.randn(B, K + 24, generator=g, device=DEV).to(torch.bfloat16)
    X = wide[:, 8:8 + K]                                     # rows apart, 16-byte aligned
    Y = _call(dq, w, X)
    _status_ok(dq)
    _check(Y, X, Wd, f"{N}x{K} batch {B}")
    assert torch.equal(Y, _call(dq, w, X))


@pytest.mark.parametrize("csize", range(1, 9))
@pytest.mark.parametrize("N,K", [(300 // 16 * 16, 2304), (1024, 4096), (2048, 640)])
def test_fp4_decode_every_cluster_size(dq, N, K, csize):  # noqa: F811
    g, w, Wd = _pack(dq, N, K, 5)
    X = torch.randn(3, K, generator=g, device=DEV).to(torch.bfloat16)
    steps = (K + 255) // 256
    if csize > steps:
        with pytest.raises(dq.DQError):
            dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=FP4, warps_per_group=csize)
        return
    Y = dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=FP4, warps_per_group=csize)
    _status_ok(dq)
    _check(Y, X, Wd, f"{csize} CTAs per tile")


@pytest.mark.parametrize("N,K", [(38160, 2304), (38160, 4352), (38160, 6400)])
def test_fp4_decode_several_tiles_and_groups_per_cta(dq, N, K):  # noqa: F811
    """More tiles than SMs and rows of two to four groups of 2048 weights, the last of them one step long: ring, accumulators and the
    groups' powers of two go on across the tiles.  A column has one large group, the others 2^30 below: the scale of another group, or of
    the next tile's, would show."""
    g, w, Wd = _pack(dq, N, K, K)
    groups = (K + 2047) // 2048
    X = torch.randn(16, K, generator=g, device=DEV)
    at = torch.arange(K, device=DEV) // 2048
    for b in range(16):
        X[b, at != b % groups] *= 2.0 ** -30
    X = X.to(torch.bfloat16)
    Yr, S = (X.double() @ Wd.T).cpu().numpy(), (X.double().abs() @ Wd.abs().T).cpu().numpy()
    for first, B in [(b, 1) for b in range(groups)] + [(0, 4), (1, 4), (0, 5), (0, 8), (3, 9), (0, 16)]:
        for _ in range(3):
            Y = _call(dq, w, X[first:first + B])
            _status_ok(dq)
            check_outputs(_f64(Y), Yr[first:first + B], S[first:first + B], f"{N}x{K}, columns {first} to {first + B - 1}")


@pytest.mark.parametrize("B", [2, 7, 12])
def test_fp4_decode_magnitudes(dq, B):  # noqa: F811
    """Rows of 40 binades; elements 2^27 below the largest of their block under a weight of zero there; subnormals; very large
    values; columns of zeros; one element alone, which is exact."""
    N, K = 272, 2560
    g, w, Wd = _pack(dq, N, K, 77)
    X = torch.zeros(B, K, dtype=torch.float32, device=DEV)
    X[0] = torch.randn(K, generator=g, device=DEV) * torch.exp2(torch.randint(-40, 1, (K,), generator=g, device=DEV).float())
    X[1, ::16] = 2.0 ** 20
    X[1, 5::16] = torch.randn(K // 16, generator=g, device=DEV).abs() * 2.0 ** -6 + 2.0 ** -7
    if B > 2:
        X[2] = torch.randint(1, 128, (K,), generator=g, device=DEV).float() * 2.0 ** -133
        X[3] = torch.randn(K, generator=g, device=DEV).sign() * 2.0 ** 104      # sums, before the tensor scale, below 2^128
        X[5, 1777] = -1.5625
        X[6] = torch.randn(K, generator=g, device=DEV)
        X[6, 2048:] *= 2.0 ** 60                              # groups of very different size
    X = X.to(torch.bfloat16)
    Y = _call(dq, w, X)
    _status_ok(dq)
    rows = [b for b in range(B) if b != 2]                    # the subnormal row's outputs are below bf16's range
    _check(Y[rows], X[rows], Wd, "magnitudes")
    if B > 2:
        assert torch.equal(Y[5], (X[5].double() @ Wd.T).to(torch.float32).to(torch.bfloat16))
        assert (Y[4] == 0).all()


@pytest.mark.parametrize("B", [1, 4, 8, 16])
@pytest.mark.parametrize("w_exp,x_exp", [(0, 116), (-60, 124), (60, 60), (100, -110), (-90, -20), (0, -100)])
def test_fp4_decode_sums_beyond_fp32_before_the_tensor_scale(dq, B, w_exp, x_exp):  # noqa: F811
    """Outputs are finite and right wherever bf16 holds them, also where sums without the tensor scale, or a group's power of two with it, are beyond
    fp32's range."""
    N, K = 272, 4352
    g = torch.Generator(device=DEV).manual_seed(B)
    w = dq.pack_weights((torch.randn(N, K, generator=g, device=DEV) * 2.0 ** (w_exp - 6)).to(torch.bfloat16), formats=dq.FMT_NVFP4)
    X = (torch.randn(B, K, generator=g, device=DEV).double() * 2.0 ** x_exp).to(torch.bfloat16)
    Y = _call(dq, w, X)
    _status_ok(dq)
    _check(Y, X, _dequantised(dq, w, "nvfp4"), f"weights 2^{w_exp - 6}, activations 2^{x_exp}")


@pytest.mark.parametrize("B", [4, 16])
def test_fp4_decode_infinities_and_nan(dq, B):  # noqa: F811
    N, K = 272, 2304
    g, w, Wd = _pack(dq, N, K, 21)
    X = torch.randn(B, K, generator=g, device=DEV).to(torch.bfloat16)
    Y0 = _call(dq, w, X)
    X[0, 700] = float("inf")
    X[1, 129], X[1, 131], X[1, 2200] = float("inf"), float("-inf"), float("-inf")
    X[2, 64] = float("nan")
    Y = _call(dq, w, X)
    _status_ok(dq)
    Yr = X.double() @ Wd.T
    for b in range(2):
        assert torch.equal(torch.isnan(Y[b]), torch.isnan(Yr[b])) and torch.equal(Y[b].double().nan_to_num(0.0, 1.0, -1.0), Yr[b].nan_to_num(0.0, 1.0, -1.0))
    assert torch.isnan(Y[2]).all()
    assert torch.equal(Y[3:], Y0[3:])


@pytest.mark.parametrize("K", [2048, 17408])
def test_fp4_decode_share_of_misrounded_outputs(dq, K):  # noqa: F811
    """As few outputs as with the kernels beside it differ from the exact sum rounded once: 0.2e-4 to 1.2e-4 measured, 1.6e-4 with the
    mma.sync kernel; 163840 outputs scatter by 0.3e-4."""
    g, w, Wd = _pack(dq, 10240, K, K)
    X = torch.randn(16, K, generator=g, device=DEV).to(torch.bfloat16)
    exact = (X.double() @ Wd.T).to(torch.float32).to(torch.bfloat16)
    for Y, n in ((_call(dq, w, X), 16), (_call(dq, w, X[:4]), 4)):
        assert float((Y != exact[:n]).double().mean()) < 3e-4
    _status_ok(dq)


def test_fp4_decode_workspace_arguments_and_graphs(dq):  # noqa: F811
    g, w, Wd = _pack(dq, 512, 512, 3)
    X = torch.randn(9, 512, generator=g, device=DEV).to(torch.bfloat16)
    need = dq.decode_nvfp4_workspace_bytes(w, 9, True)
    ws = torch.empty(need + 256, dtype=torch.uint8, device=DEV)
    with pytest.raises(dq.DQError):
        dq.decode_linear_nvfp4_ws(w, X, ws[:need - 1])
    with pytest.raises(dq.DQError):
        dq.decode_linear_nvfp4_ws(w, X, ws[16:])
    for B in (4, 17):
        with pytest.raises(dq.DQError):
            dq.decode_linear_nvfp4_ws(w, torch.zeros(B, 512, dtype=torch.bfloat16, device=DEV), ws)
    # a large matrix whose calls borrow a workspace, replayed from a graph and on several streams
    g, w, Wd = _pack(dq, 28672, 4096, 4)
    X = torch.randn(16, 4096, generator=g, device=DEV).to(torch.bfloat16)
    assert dq.decode_nvfp4_workspace_bytes(w, 16) > 0 and dq.decode_nvfp4_workspace_bytes(w, 4) == 0
    Y0 = dq.decode_linear_nvfp4(w, X)
    out = torch.empty_like(Y0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(3):
            dq.decode_linear_nvfp4(w, X, out=out)
    for _ in range(3):
        out.zero_()
        graph.replay()
        assert torch.equal(out, Y0)
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    outs = []
    for i in range(9):
        with torch.cuda.stream(streams[i % 3]):
            outs.append(dq.decode_linear_nvfp4(w, X[:5 + i % 3 * 4]))
    torch.cuda.synchronize()
    other = dq.decode_linear_nvfp4(w, X, stream=streams[0])  # another stream than the current one: it is borrowed there
    torch.cuda.synchronize()
    _status_ok(dq)
    _check(other, X, Wd, "explicit stream")
    for i, Y in enumerate(outs):
        n = 5 + i % 3 * 4
        assert torch.equal(Y, outs[i % 3]) and Y.shape[0] == n
        _check(Y, X[:n], Wd, f"stream {i % 3}")


class _ForeignStream:
    def __init__(self, cuda_stream):
        self.cuda_stream = cuda_stream


def test_fp4_decode_same_bits_on_every_stream(dq):  # noqa: F811
    """A call gives the same bits on the current stream, on another of torch's, on one that torch knows by its address alone and on the
    default one; what it borrows belongs to the stream that it runs on."""
    g, w, Wd = _pack(dq, 28672, 4096, 8)
    assert dq.decode_nvfp4_workspace_bytes(w, 8) > 0
    X = torch.randn(8, 4096, generator=g, device=DEV).to(torch.bfloat16)
    Y0 = dq.decode_linear_nvfp4(w, X)
    assert not torch.equal(Y0, dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=5)) and not torch.equal(Y0, dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=6))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    outs = []
    for _ in range(4):
        for s in (side, _ForeignStream(side.cuda_stream), _ForeignStream(0), torch.cuda.default_stream()):
            outs.append(dq.decode_linear_nvfp4(w, X, stream=s))
        with torch.cuda.stream(side):
            outs.append(dq.decode_linear_nvfp4(w, X, stream=_ForeignStream(0)))
            outs.append(dq.decode_linear_nvfp4(w, X))
    torch.cuda.synchronize()
    _status_ok(dq)
    for Y in outs:
        assert torch.equal(Y, Y0)


def test_fp4_decode_captures_that_torch_does_not_know_of(dq):  # noqa: F811
    """A graph captured without torch keeps no hold on torch's memory: a call with `out` given may leave nothing of torch's in it.  Whatever
    torch hands out afterwards stays as it is while the graph is replayed.  (In torch's own captures the workspace is the graph's.)"""
    runtime = pytest.importorskip("cuda.bindings.runtime")
    g, w, Wd = _pack(dq, 28672, 4096, 8)
    X = torch.randn(8, 4096, generator=g, device=DEV).to(torch.bfloat16)
    need = dq.decode_nvfp4_workspace_bytes(w, 8)
    assert need > 0
    out = torch.empty(8, 28672, dtype=torch.bfloat16, device=DEV)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for warm in (True, False):                               # with a free block of that size in torch's hands, and with nothing
        torch.cuda.empty_cache()
        with torch.cuda.stream(side):
            if warm:
                torch.empty(need, dtype=torch.uint8, device=DEV)
            ok, = runtime.cudaStreamBeginCapture(side.cuda_stream, runtime.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal)
            assert int(ok) == 0
            dq.decode_linear_nvfp4(w, X, out=out)
            ok, graph = runtime.cudaStreamEndCapture(side.cuda_stream)
            assert int(ok) == 0
            ok, exe = runtime.cudaGraphInstantiate(graph, 0)
            assert int(ok) == 0
            others = [torch.full((need,), 171, dtype=torch.uint8, device=DEV) for _ in range(4)]
            out.zero_()
            for _ in range(2):
                ok, = runtime.cudaGraphLaunch(exe, side.cuda_stream)
                assert int(ok) == 0
        side.synchronize()
        _status_ok(dq)
        assert all(bool((t == 171).all()) for t in others)
        _check(out, X, Wd, "replayed")
        assert int(runtime.cudaGraphExecDestroy(exe)[0]) == 0 and int(runtime.cudaGraphDestroy(graph)[0]) == 0
    # torch's own capture: the kernel with a workspace, which stays the graph's
    Y0 = dq.decode_linear_nvfp4(w, X)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dq.decode_linear_nvfp4(w, X, out=out)
    others = [torch.full((need,), 171, dtype=torch.uint8, device=DEV) for _ in range(4)]
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, Y0) and all(bool((t == 171).all()) for t in others)


def test_fp4_decode_workspace_is_memory_of_its_size(dq):  # noqa: F811
    """A workspace whose elements do not lie one after the other, or that is not on the GPU, is refused; its size counts in bytes."""
    g, w, Wd = _pack(dq, 512, 512, 3)
    X = torch.randn(9, 512, generator=g, device=DEV).to(torch.bfloat16)
    need = dq.decode_nvfp4_workspace_bytes(w, 9, True)
    for ws in (torch.empty(1, dtype=torch.uint8, device=DEV).expand(need), torch.empty(2 * need, dtype=torch.uint8, device=DEV)[::2],
               torch.empty(need, dtype=torch.uint8)):
        with pytest.raises(AssertionError):
            dq.decode_linear_nvfp4_ws(w, X, ws)
    _check(dq.decode_linear_nvfp4_ws(w, X, torch.empty((need + 3) // 4, dtype=torch.float32, device=DEV)), X, Wd, "fp32 workspace")


@pytest.mark.parametrize("B", [5, 8, 9, 13, 16])
@pytest.mark.parametrize("tiles", [74, 68, 49, 45, 36, 29, 24, 21, 18, 9])
def test_fp4_decode_clusters_with_a_workspace(dq, tiles, B):  # noqa: F811
    """Clusters of every size that tiles of these numbers can share, with one and with two times four columns to add up for each CTA of a
    cluster, and groups that a CTA's share of the row cuts."""
    for K in (2304, 4352):
        N = tiles * 256 - 112
        g, w, Wd = _pack(dq, N, K, tiles)
        X = torch.randn(B, K, generator=g, device=DEV).to(torch.bfloat16)
        Y = _call(dq, w, X)
        _status_ok(dq)
        _check(Y, X, Wd, f"{N}x{K} batch {B}")
        assert torch.equal(Y, _call(dq, w, X))


@pytest.mark.parametrize("B", [4, 16])
@pytest.mark.parametrize("K", [2048, 16384])
def test_fp4_decode_digits_larger_than_their_sum(dq, K, B):  # noqa: F811
    """Activations just above half a digit beside larger ones, so that a value's digits add up to three times its magnitude, with sums that
    cancel: inside the allowance of the other kernels, and no worse than the mma.sync and the batch kernel (2.9e-8 to 7.4e-8 of the sum of
    magnitudes beyond the rounding to bf16, for 0 to 1.2e-7 of theirs)."""
    N = 1024
    g = torch.Generator(device=DEV).manual_seed(K)
    half = (torch.randn(N, K // 2, generator=g, device=DEV) * 0.02).abs()
    w = dq.pack_weights(torch.cat((half, -half), dim=1).to(torch.bfloat16), formats=dq.FMT_NVFP4)
    Wd = _dequantised(dq, w, "nvfp4")
    x = 0.5 + 2.0 ** -8 * torch.randint(1, 4, (B, K // 2), generator=g, device=DEV).float()
    x[:, ::16] = 3.0
    X = torch.cat((x, x), dim=1)
    X[:, K // 2 + 5::16] += 2.0 ** -8                       # leaves a small sum
    X = X.to(torch.bfloat16)
    Y = _call(dq, w, X)
    _status_ok(dq)
    Yr, S = X.double() @ Wd.T, X.double().abs() @ Wd.abs().T
    assert float((Yr.abs() / S).max()) < 1e-2               # they do cancel
    ulp = torch.exp2(torch.floor(torch.log2(Yr.abs().clamp_min(2.0 ** -126))) - 7)
    over = ((Y.double() - Yr).abs() - 0.5 * ulp) / S
    assert float(over.max()) < 3e-7                         # four times the most that was seen


@pytest.mark.parametrize("N,K,csize", [(1024, 4096, 1), (1024, 4096, 4), (40000, 512, 0)])
@pytest.mark.parametrize("B", [1, 4])
def test_fp4_decode_wait_runs_out(dq, N, K, csize, B):  # noqa: F811
    """Weights that are never requested: the waits run out in every role, the clusters' barriers are met, the launch returns and reports, and
    the next call is right."""
    g, w, Wd = _pack(dq, N, K, 9)
    X = torch.randn(B, K, generator=g, device=DEV).to(torch.bfloat16)
    good = dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=FP4, warps_per_group=csize)
    dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=9, warps_per_group=csize, wait_cycles=2_000_000)
    torch.cuda.synchronize()
    st, _ = dq.get_status()
    assert dq.status_string(st) == "device-side wait ran out"
    assert torch.equal(dq.test_decode_linear(w, dq.FMT_NVFP4, X, variant=FP4, warps_per_group=csize, wait_cycles=2_000_000), good)
    _status_ok(dq)
