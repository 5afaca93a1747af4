"""The GEMM with the weights on the M side of the MMA, at the edges of its tiles, and the merge of the LM head's records, at the
edges of the blocks of rows a warp takes; against the oracle's functions."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import l2pd_oracle as orc
from paper_2509_25188_b200 import workloads as wl

pytestmark = pytest.mark.gpu

WM = 10_000_000   # tile code: weights on the M side; the width is the rows of a tile


def _bf16(seed, stream, shape, std):
    return wl.make_activations(seed, stream, shape, std, "bf16")


def _close_bf16(got, want, sums):
    # fp32 sums of K exact products, K 2^-24 of the sum of magnitudes at most, then one rounding to bf16 (2^-9, twice for the
    # two roundings of a SwiGLU's factors in fp32 arithmetic of a few ulp)
    assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + sums).all()


@pytest.mark.parametrize("M,N,K,tile", [(1, 128, 64, 1032), (15, 104, 72, 1032), (17, 256, 1032, 1032), (128, 136, 192, 1128),
                                        (129, 520, 320, 1144), (257, 1040, 136, 2144), (300, 528, 1032, 2112), (513, 264, 512, 2256),
                                        (1029, 2064, 320, 2176), (700, 1536, 128, 1064)])
def test_gemm_with_rows_on_the_n_side(M, N, K, tile):
    """One row, tiles with a ragged last chunk, several row tiles per weight tile, weight tiles with a ragged end, single CTAs and
    pairs (the second CTA without features too), a K tail; gate and up matrices in either order of address."""
    from paper_2509_25188_b200 import binding as b
    A, W, W2 = _bf16(11, 0, (M, K), 1.0), _bf16(11, 1, (N, K), 0.05), _bf16(11, 2, (N, K), 0.05)
    a, w, w2 = orc.widen(A), orc.widen(W), orc.widen(W2)
    dA, dW, dW2 = b.to_device(A), b.to_device(W), b.to_device(W2)
    want, up = orc.linear(a, W), orc.linear(a, W2)
    mag, mag2 = np.abs(a) @ np.abs(w).T, np.abs(a) @ np.abs(w2).T
    eps = (K + 4) * 2.0 ** -24
    _close_bf16(b.gemm_bf16(dA, dW, WM + tile).float().cpu().numpy(), want, eps * mag)
    # |silu'| < 1.1, so an error of the gate's sum moves the result by 1.1 |up| of it
    for g, u, gm, um, dg, du in ((want, up, mag, mag2, dW, dW2), (up, want, mag2, mag, dW2, dW)):
        _close_bf16(b.gemm_bf16_swiglu(dA, dg, du, WM + tile).float().cpu().numpy(), orc.silu(g) * u,
                    eps * (1.1 * np.abs(u) * gm + np.abs(g) * um) + 2.0 ** -20 * np.abs(g * u))
    X = wl.make_activations(11, 3, (M, N), 1.0, "fp32")
    got = b.gemm_bf16_residual(dA, dW, b.to_device(X.copy()), WM + 10000 + tile).cpu().numpy()
    assert (np.abs(got - (X.astype(np.float64) + want)) <= eps * (mag + np.abs(X))).all()


@pytest.mark.parametrize("M,N,K,slices", [(1, 128, 1024, 4), (3, 520, 1032, 2), (5, 520, 4104, 4), (32, 4096, 2048, 4), (97, 1000, 1024, 2),
                                          (125, 4096, 1024, 4), (128, 512, 2048, 4)])
def test_k_slices_of_a_cluster(M, N, K, slices):
    """Slices that meet in shared memory: CTAs without rows of their own, uneven shares, a ragged feature tile, a shorter last
    slice.  The sum is taken in slice order, so that it repeats bit for bit."""
    from paper_2509_25188_b200 import binding as b
    A, W = _bf16(12, 0, (M, K), 1.0), _bf16(12, 1, (N, K), 0.05)
    X = wl.make_activations(12, 2, (M, N), 1.0, "fp32")
    a, dA, dW = orc.widen(A), b.to_device(A), b.to_device(W)
    code = WM + 10000 * slices + 1000 + max(32, (M + 15) // 16 * 16)
    got = [b.gemm_bf16_residual(dA, dW, b.to_device(X.copy()), code).cpu().numpy() for _ in range(2)]
    bound = (K + 4) * 2.0 ** -24 * (np.abs(a) @ np.abs(orc.widen(W)).T + np.abs(X))
    assert (np.abs(got[0] - (X.astype(np.float64) + orc.linear(a, W))) <= bound).all()
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("block,vocab", [(1, 2000), (15, 2000), (16, 70), (17, 5000), (33, 2000), (64, 20000)])
def test_merge_of_the_records_of_a_block(block, vocab):
    """Fewer and more records than warps, one and several blocks of rows, the last of them ragged."""
    from paper_2509_25188_b200 import binding as b
    shape = wl.ModelShape(n_layers=1, d_model=128, n_heads=1, head_dim=128, d_ff=256, vocab=vocab, rms_eps=1e-5, rope_theta=10000.0,
                          mask_id=vocab - 1, eot_id=vocab - 2, dtype="bf16")
    dec = b.Decoder(shape, wl.make_weights(shape, seed=3, final_norm_gain=wl.spread_gain(shape)), None, block_len=block, max_batch=3,
                    max_seq=7 + block, use_filter=False)
    dec.state_reset(wl.make_prompts(3, 7, shape, seed=2), block)
    out = dec.denoise_step(want_logits=True)
    dec.close()
    pred, conf, _ = orc.confidence_head(out["logits"].reshape(3 * block, vocab).astype(np.float64))
    assert np.array_equal(out["pred"].reshape(-1), pred)
    # sums of `vocab` exponentials in fp32, each a few ulp
    assert np.abs(out["conf"].reshape(-1) - conf).max() <= 1e-5


@pytest.mark.parametrize("code,residual,M,N,K", [
    (WM + 30000, True, 64, 512, 2048),               # three slices
    (WM + 80000, True, 64, 512, 2048),               # eight
    (WM + 42000, True, 64, 512, 2048),               # four slices on pairs
    (WM + 40000 + 1144, True, 300, 512, 2048),       # four slices of tiles of 144 rows
    (WM + 40000 + 1064, True, 64, 128 * 200, 2048),  # more slices than SMs
    (WM + 200000, False, 300, 512, 512),             # two slabs of rows, which the weights' side has not
    (WM + 1000000, False, 300, 512, 512),            # two issuing threads, neither
    (3 * WM, False, 300, 512, 512),                  # no such orientation
    (9 * WM + 2128, False, 300, 512, 512)])
def test_unsupported_tile_codes_are_refused(code, residual, M, N, K):
    """L2PD_ERR_SHAPE, nothing launched and nothing written."""
    import torch
    from paper_2509_25188_b200 import binding as b
    A, W = torch.ones(M, K, dtype=torch.bfloat16, device="cuda"), torch.ones(N, K, dtype=torch.bfloat16, device="cuda")
    X = torch.zeros(M, N, device="cuda")
    with pytest.raises(b.L2pdError) as e:
        b.gemm_bf16_residual(A, W, X, code) if residual else b.gemm_bf16(A, W, code)
    assert e.value.status == -2
    assert not X.any()


@pytest.mark.parametrize("code,M", [(WM + 40000, 64), (WM + 20000, 300), (WM + 40000, 200), (WM + 100000 + 2000000, 300)])
def test_tile_codes_that_leave_parts_open(code, M):
    """Slices with the tile left open get single CTAs and a tile that their exchange has room for; one slab and no second issuer is
    what this side has."""
    from paper_2509_25188_b200 import binding as b
    N, K = 512, 2048
    A, W, X = _bf16(13, 0, (M, K), 1.0), _bf16(13, 1, (N, K), 0.05), wl.make_activations(13, 2, (M, N), 1.0, "fp32")
    a = orc.widen(A)
    got = b.gemm_bf16_residual(b.to_device(A), b.to_device(W), b.to_device(X.copy()), code).cpu().numpy()
    bound = (K + 4) * 2.0 ** -24 * (np.abs(a) @ np.abs(orc.widen(W)).T + np.abs(X))
    assert (np.abs(got - (X.astype(np.float64) + orc.linear(a, W))) <= bound).all()


def _kernels(call):
    """Names of the kernels that call() launches, from a capture of it (the driver's own account of the graph's nodes)."""
    import ctypes as C
    import torch

    class Node(C.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
        _fields_ = [("func", C.c_void_p), ("dims", C.c_uint * 7), ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]

    cu = C.CDLL("libcuda.so.1")
    call()                     # what a first call sets up is not capturable
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw, n, names = C.c_void_p(graph.raw_cuda_graph()), C.c_size_t(), []
    assert cu.cuGraphGetNodes(raw, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(raw, nodes, C.byref(n)) == 0
    for node in nodes:
        kind, p, name = C.c_int(), Node(), C.c_char_p()
        assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        if kind.value == 0:    # a kernel
            assert cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)) == 0
            f = cu.cuFuncGetName(C.byref(name), C.c_void_p(p.func)) if p.func else cu.cuKernelGetName(C.byref(name), C.c_void_p(p.kern))
            assert f == 0
            names.append(name.value.decode())
    return names


@pytest.mark.parametrize("epi,M,N,K,m_side", [
    ("res", 160, 4096, 4096, False), ("res", 256, 2048, 2048, False), ("store", 64, 3072, 1024, False),   # few rows
    ("res", 300, 1024, 2816, False),                                                                    # no slices unasked
    ("store", 300, 1536, 512, False), ("swiglu", 257, 1376, 512, False),                                # few k-blocks
    ("store", 1029, 12288, 4096, True), ("res", 1029, 2048, 5632, True), ("swiglu", 400, 12288, 4096, True)])
def test_automatic_calls_take_the_faster_side(epi, M, N, K, m_side):
    """us, rows on the M side and weights there: 160 x 4096 x 4096 11.8 and 14.3, 256 x 2048 x 2048 9.8 and 16.0, 64 x 3072 x 1024 5.9 and
    6.6, 300 x 1024 x 2816 6.8 and 10.6, 300 x 1536 x 512 5.3 and 5.8, 257 x 1376 x 512 5.4 and 6.0; 1029 x 12288 x 4096 100 and 83, 1029 x 2048
    x 5632 23.8 and 21.4, 400 x 12288 x 4096 (SwiGLU) 93 and 82."""
    import torch
    from paper_2509_25188_b200 import binding as b
    A, W, U = (torch.zeros(r, K, dtype=torch.bfloat16, device="cuda") for r in (M, N, N))
    X, C = torch.zeros(M, N, device="cuda"), torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")

    def call():
        s = torch.cuda.current_stream().cuda_stream
        if epi == "res":
            r = b.lib.l2pd_gemm_bf16_residual(s, A.data_ptr(), W.data_ptr(), X.data_ptr(), M, N, K, 0, 0)
        elif epi == "swiglu":
            r = b.lib.l2pd_gemm_bf16_swiglu(s, A.data_ptr(), W.data_ptr(), U.data_ptr(), C.data_ptr(), M, N, K, 0, 0)
        else:
            r = b.lib.l2pd_gemm_bf16(s, A.data_ptr(), W.data_ptr(), C.data_ptr(), M, N, K, 0, 0)
        assert r == 0
    names = _kernels(call)
    assert len(names) == 1 and ("gemm_wm" in names[0]) == m_side, names
