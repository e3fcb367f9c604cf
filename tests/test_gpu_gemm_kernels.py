"""GPU parity of every prefill GEMM kernel and split, forced through the test hook: CTA pairs, lone CTAs and clusters on tiles of 128 and
256 columns, columns shared out over two launches.  Against the CPU oracle at sizes that end inside a tile, a k-step and a 32-row
quarter, with the tolerances of parity_utils."""
import numpy as np
import pytest
import torch

import dq_inputs
from parity_utils import check_outputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PAIR, TILES128, TILES256, TWO_LAUNCHES = 1, 2, 3, 4


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


def _call(oracle, M, N, K):
    """Weights, activations and the oracle's result for them."""
    if (M, N, K) not in _cache:
        W = dq_inputs.gaussian_bf16(N, K, 0.02, 600 + N + K)
        A = dq_inputs.gaussian_bf16(M, K, 1.0, 601 + M)
        sa = dq_inputs.static_act_scale(A)
        ref = oracle.pack_weights(dq_inputs.bf16_to_f32_numpy(W))
        Yr, S = oracle.prefill_linear(dq_inputs.bf16_to_f32_numpy(A), sa, ref["nvfp4_codes"], ref["nvfp4_scales"], ref["s"])
        _cache[(M, N, K)] = (W, A, sa, Yr, S)
    return _cache[(M, N, K)]


# (M, N, K): rows and columns that end inside a tile of 128 or 256, K that ends inside a k-step of 256, several row and column tiles
SHAPES = [(1, 256, 128), (77, 272, 640), (129, 272, 1152), (200, 528, 384), (300, 784, 640), (513, 1040, 1408), (640, 1536, 2048),
          (260, 16, 2176), (385, 400, 256)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_every_gemm_kernel(dq, oracle, M, N, K):
    W, A, sa, Yr, S = _call(oracle, M, N, K)
    w = dq.pack_weights(W.to(DEV), formats=dq.FMT_NVFP4)
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w, M), DEV)
    dq.prefill_quantize(w, A.to(DEV), sa, ws)
    steps = (K + 255) // 256
    for kernel, bn in ((PAIR, 0), (TILES128, 128), (TILES256, 256), (TWO_LAUNCHES, 128)):
        for c in (1,) if kernel == PAIR else range(1, 9):
            out = torch.full((M + 1, N + 16), 7.0, dtype=torch.bfloat16, device=DEV)           # guarded, strided
            cols = N if kernel != TWO_LAUNCHES else N - (N - 1) // 256 * 256                   # what the clusters take
            tiles = -(-M // 128) * -(-cols // bn) if bn else 0
            if (kernel == TWO_LAUNCHES and N <= 256) or c > steps or tiles * c > 148:
                with pytest.raises(dq.DQError) as e:
                    dq.test_prefill_gemm(w, M, sa, out[:M, :N], ws, kernel, c)
                assert e.value.code == 1
                continue
            try:
                dq.test_prefill_gemm(w, M, sa, out[:M, :N], ws, kernel, c)
            except dq.DQError as e:                                    # clusters do not straddle the GPU's groups of SMs: fewer may fit
                assert e.code == 1 and tiles * c > 100
                continue
            _status_ok(dq)
            check_outputs(out[:M, :N].float().cpu().numpy().astype(np.float64), Yr, S, f"kernel {kernel}, {c} CTAs a tile, {M}x{N}x{K}")
            assert torch.all(out[M] == 7.0) and torch.all(out[:, N:] == 7.0)


@pytest.mark.parametrize("M,N,K", [(300, 784, 4736), (129, 272, 8192)])
def test_lone_ctas_and_pairs_add_up_alike(dq, M, N, K):
    """One CTA a tile adds k-step after k-step, as the pairs do: the same bits on operands whose sums depend on the order; a cluster's sums
    are in the order of its ranks and the same on every call."""
    g = torch.Generator(device=DEV).manual_seed(M)

    def wide(rows, std):
        e = torch.randint(-9, 1, (rows, K // 16), generator=g, device=DEV).float()
        return (torch.randn(rows, K, generator=g, device=DEV) * std * torch.exp2(e).repeat_interleave(16, 1)).to(torch.bfloat16)

    w = dq.pack_weights(wide(N, 0.02), formats=dq.FMT_NVFP4)
    A = wide(M, 1.0)
    sa = float(A.abs().max()) / 2688.0
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w, M), DEV)
    dq.prefill_quantize(w, A, sa, ws)
    run = lambda kernel, c=0: dq.test_prefill_gemm(w, M, sa, torch.empty(M, N, dtype=torch.bfloat16, device=DEV), ws, kernel, c)
    want = run(PAIR)
    for kernel in (TILES128, TILES256, TWO_LAUNCHES):
        assert torch.equal(run(kernel), want), f"kernel {kernel}"
    assert torch.equal(run(TILES128, 4), run(TILES128, 4)) and torch.equal(run(TILES128, 4), run(TILES256, 4))
    _status_ok(dq)


@pytest.mark.parametrize("kernel,c", [(PAIR, 0), (TILES128, 0), (TILES128, 4), (TILES256, 3), (TWO_LAUNCHES, 2)])
def test_gemm_kernels_replay_from_a_cuda_graph(dq, kernel, c):
    """Quantiser and GEMM, captured: replays on new activations give what eager calls give."""
    M, N, K = 300, 784, 1152
    w = dq.pack_weights(dq_inputs.gaussian_bf16(N, K, 0.02, 650).to(DEV), formats=dq.FMT_NVFP4)
    A = dq_inputs.gaussian_bf16(M, K, 1.0, 651).to(DEV)
    sa = 5.0 / 2688.0
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w, M), DEV)
    Y = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)

    def call():
        dq.prefill_quantize(w, A, sa, ws)
        dq.test_prefill_gemm(w, M, sa, Y, ws, kernel, c)

    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for seed in (652, 653):
        A.copy_(dq_inputs.gaussian_bf16(M, K, 1.0, seed).to(DEV))
        Y.zero_()
        graph.replay()
        torch.cuda.synchronize()
        got = Y.clone()
        call()
        _status_ok(dq)
        assert torch.equal(got, Y) and float(got.float().abs().max()) > 0.0


def test_gemm_hook_arguments(dq):
    M, N, K = 64, 256, 256
    w = dq.pack_weights(dq_inputs.gaussian_bf16(N, K, 0.02, 660).to(DEV), formats=dq.FMT_NVFP4)
    ws = dq.alloc_workspace(dq.prefill_workspace_bytes(w, M), DEV)
    Y = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
    for kernel, c in ((0, 0), (5, 0), (-1, 0), (TILES128, 9), (TILES128, -1), (TILES128, 2), (TWO_LAUNCHES, 0)):
        with pytest.raises(dq.DQError) as e:
            dq.test_prefill_gemm(w, M, 1.0, Y, ws, kernel, c)
        assert e.value.code == 1
    _status_ok(dq)
