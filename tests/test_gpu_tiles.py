"""GPU parity at the edges of the persistent GEMM's and the streaming attention's
tiles: token tiles of 32 to 256 rows and their remainders, odd k-block counts,
in-CTA K chunks, the resident token tile, SwiGLU gates outside the fast
quotient's range; attention launches of more than one wave with one item, more
than eight items, windows of one row and sub-blocks of two rows.

References and tolerances as in test_gpu_kernels.py (fp32 matmul of the same
fp16 operands, 2^-11 relative for fp16 stores; the oracle's float64 softmax)."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

import synth
from oracle import decode as od
from paper_2609_26638_gb300 import build
from tests.test_gpu_kernels import DEV, _linear, _oracle_attn, _paged, _run_attention

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    from paper_2609_26638_gb300 import gs as binding
    return binding


@pytest.mark.parametrize("M,N,K,split", [
    (1, 128, 64, 1), (65, 256, 64, 1), (96, 384, 192, 3), (97, 2048, 1024, 8), (144, 1024, 704, 1),
    (145, 1024, 4096, 8), (192, 8192, 320, 1), (193, 2048, 640, 5), (256, 20480, 128, 2),
    (257, 4096, 192, 1), (1000, 1024, 1024, 16),
])
def test_linear_tile_edges(gs, M, N, K, split):
    g = torch.Generator(device=DEV).manual_seed(M + N + K)
    x = torch.randn(M, K, device=DEV, generator=g).half()
    w = (0.02 * torch.randn(N, K, device=DEV, generator=g)).half()
    ref = x.float() @ w.float().T
    y = torch.zeros(M, N, dtype=torch.float16, device=DEV)
    _linear(gs, x, w, M, N, K, gs.EPI_STORE_F16, split, y)
    torch.testing.assert_close(y.float(), ref, rtol=2e-3, atol=1e-3 * ref.abs().max().item())
    base = torch.randn(M, N, device=DEV, generator=g)
    r = base.clone()
    _linear(gs, x, w, M, N, K, gs.EPI_RESID_F32, split, r)
    torch.testing.assert_close(r, base + ref, rtol=1e-4, atol=1e-4 * ref.abs().max().item())


@pytest.mark.parametrize("M", [1, 32, 33, 300])
@pytest.mark.parametrize("K", [64, 960, 1024, 2048])
def test_linear_argmax_more_tiles_than_sms(gs, M, K):
    """153 feature tiles: with at most 32 rows and K <= 1024 the token tile stays
    resident.  The returned row is the reference's, or within the fp32 summation
    error of its value (K products of N(0, 1) x 0.02 N(0, 1), 2^-24 each)."""
    V = 153 * 128
    g = torch.Generator(device=DEV).manual_seed(M * 3 + K)
    x = torch.randn(M, K, device=DEV, generator=g).half()
    w = (0.02 * torch.randn(V, K, device=DEV, generator=g)).half()
    ref = x.double() @ w.double().T
    keys = torch.zeros(M, dtype=torch.int64, device=DEV)
    _linear(gs, x, w, M, V, K, gs.EPI_ARGMAX, 1, keys)
    idx = 0xFFFFFFFF - (keys & 0xFFFFFFFF)
    got = ref.gather(1, idx[:, None])[:, 0]
    assert bool((ref.max(dim=1).values - got <= 1e-4).all())


@pytest.mark.parametrize("M,split", [(3, 1), (40, 2), (200, 1)])
def test_swiglu_gates_of_any_size(gs, M, split):
    """Gates from about -300 to 300: exp overflows on the negative side (silu is
    then -0), and rows of zeros keep zero."""
    F, K = 512, 256
    g = torch.Generator(device=DEV).manual_seed(9 + M)
    x = torch.randn(M, K, device=DEV, generator=g).half()
    x[M // 2] = 0
    wg = torch.randn(F, K, device=DEV, generator=g) * 5.0
    wu = torch.randn(F, K, device=DEV, generator=g) * 0.02
    w = torch.cat([wg, wu]).half()
    gu = x.double() @ w.double().T
    ref = gu[:, :F] * torch.sigmoid(gu[:, :F]) * gu[:, F:]
    y = torch.full((M, F), 7.0, dtype=torch.float16, device=DEV)
    _linear(gs, x, w, M, F, K, gs.EPI_SWIGLU, split, y)
    torch.testing.assert_close(y.double(), ref, rtol=2e-3, atol=1e-3)
    assert float(y[M // 2].abs().max()) == 0.0


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("B,W,lo,hi,Hq,Hkv,sp", [
    (40, 1, 1, 200, 16, 8, 4),       # rows of one token: two per block
    (24, 17, 30, 900, 16, 8, 1),     # up to fifteen items, merged through scratch
    (6, 65, 500, 1400, 16, 8, 3),    # sub-blocks of 128 and of 2 rows
    (80, 9, 0, 60, 4, 4, 2),         # one item per sequence
])
def test_attention_streams_items(gs, mode, B, W, lo, hi, Hq, Hkv, sp):
    rng = np.random.default_rng(B + W + mode)
    ns = [int(v) for v in rng.integers(lo, hi + 1, B)]
    q, k, v = synth.attn_inputs(B, W, hi + W + 1, Hq, Hkv, index=B + mode)
    pool, pt, _ = _paged(k, v, rng)
    got = _run_attention(gs, mode, q, pool, pt, np.array(ns), W, Hq, Hkv, sp)
    K = W - 1
    for b in sorted({0, B - 1, int(np.argmax(ns)), int(np.argmin(ns))}):
        allowed = od.draft_allowed(ns[b], K) if mode == 0 else od.verify_allowed(ns[b], K)
        nk = allowed.shape[1]
        want = _oracle_attn(q[b].astype(np.float64), k[b, :nk].astype(np.float64),
                            v[b, :nk].astype(np.float64), allowed, Hq, Hkv)
        np.testing.assert_allclose(got[b], want, rtol=5e-3, atol=5e-3)


_SILU_CHECK = r"""
#include "gemm_tc.cuh"
__device__ unsigned long long n_bad;
__device__ unsigned first_bad = 0xFFFFFFFFu;
// every float bit pattern in [lo, hi]
__global__ void check(unsigned lo, unsigned hi) {
  const unsigned long long step = 1ull * gridDim.x * blockDim.x;
  for (unsigned long long u = lo + 1ull * blockIdx.x * blockDim.x + threadIdx.x; u <= hi; u += step) {
    const float g = __uint_as_float(static_cast<unsigned>(u));
    if (__float_as_uint(gs::silu_in_range(g)) != __float_as_uint(gs::silu_any(g))) {
      atomicAdd(&n_bad, 1ull);
      atomicMin(&first_bad, static_cast<unsigned>(u));
    }
  }
}
extern "C" int silu_check(unsigned long long* bad, unsigned* first) {
  check<<<1216, 256>>>(0u, 0x7149F2CAu);            // +0 .. 1e30
  check<<<1216, 256>>>(0x80000000u, 0xC2AA0000u);   // -0 .. -85
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  return cudaMemcpyFromSymbol(bad, n_bad, 8) != cudaSuccess ||
         cudaMemcpyFromSymbol(first, first_bad, 4) != cudaSuccess;
}
"""


def test_silu_quotient_equals_the_division_in_every_bit(tmp_path):
    """silu_in_range against g / (1 + __expf(-g)) for every float of its range,
    denormals and both zeros included, built with the library's own flags."""
    assert np.float32(1e30).view(np.uint32) == 0x7149F2CA
    assert np.float32(-85.0).view(np.uint32) == 0xC2AA0000
    src, lib = tmp_path / "silu_check.cu", tmp_path / "silu_check.so"
    src.write_text(_SILU_CHECK)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src),
                    "-o", str(lib)], check=True)
    bad, first = ctypes.c_ulonglong(), ctypes.c_uint()
    assert ctypes.CDLL(str(lib)).silu_check(ctypes.byref(bad), ctypes.byref(first)) == 0
    assert bad.value == 0, f"{bad.value} floats differ, the first is 0x{first.value:08X}"


@pytest.mark.parametrize("B,W,Hq,Hkv,sp,n", [
    (4, 65, 16, 8, 2, 700),        # 4 x 2 x 8 x 6 = 384 CTAs in clusters, blocks of 128 and 2 rows
    (3, 97, 16, 8, 2, 400),        # 4 items: 192 CTAs, one wave
    (14, 17, 16, 2, 3, 1200),      # 14 x 2 x 2 x 7 = 392 CTAs, blocks of 128 and 8 rows
])
def test_attention_clusters_of_two_waves(gs, B, W, Hq, Hkv, sp, n):
    """Blocks of more than 96 rows in clusters of up to eight items, one to two
    waves of CTAs: the same rows as each sequence's own launch (one wave), and the
    oracle's masked softmax."""
    rng = np.random.default_rng(B)
    ns = [n - 37 * b for b in range(B)]
    q, k, v = synth.attn_inputs(B, W, n + W + 1, Hq, Hkv, index=B)
    pool, pt, _ = _paged(k, v, rng)
    got = _run_attention(gs, 1, q, pool, pt, np.array(ns), W, Hq, Hkv, sp)
    for b in (0, B - 1):
        one = _run_attention(gs, 1, q[b:b + 1], pool, pt[b:b + 1], np.array(ns[b:b + 1]), W, Hq, Hkv, sp)
        assert np.array_equal(got[b], one[0])
        allowed = od.verify_allowed(ns[b], W - 1)
        nk = allowed.shape[1]
        want = _oracle_attn(q[b].astype(np.float64), k[b, :nk].astype(np.float64),
                            v[b, :nk].astype(np.float64), allowed, Hq, Hkv)
        np.testing.assert_allclose(got[b], want, rtol=5e-3, atol=5e-3)


@pytest.mark.parametrize("N,K,Ms", [(1024, 4096, (65, 128, 129, 256, 257, 320)),
                                    (2048, 8192, (65, 128, 129)), (256, 4096, (65, 600, 1216, 1217))])
def test_clusters_above_64_rows(gs, N, K, Ms):
    """Splits of eight over windows of more than 64 rows, on both sides of the
    launch size up to which they run as clusters (304 CTAs): the first rows' bits
    are those of a 17-row window, the result is the fp32 matmul's, and a scratch
    of the stated size full of stale bytes serves, its error word left at zero."""
    g = torch.Generator(device=DEV).manual_seed(N + K)
    x = torch.randn(max(Ms), K, device=DEV, generator=g).half()
    w = (0.02 * torch.randn(N, K, device=DEV, generator=g)).half()
    base = torch.randn(max(Ms), N, device=DEV, generator=g)
    few = base[:17].clone()
    _linear(gs, x[:17].contiguous(), w, 17, N, K, gs.EPI_RESID_F32, 8, few)
    for M in Ms:
        xm = x[:M].contiguous()
        y = base[:M].clone()
        sb = gs.gs_linear_scratch_bytes(M, N, 8)
        scratch = torch.full((sb,), 0x7F, dtype=torch.uint8, device=DEV)
        gs.gs_linear(xm.data_ptr(), w.data_ptr(), y.data_ptr(), M, N, K, gs.EPI_RESID_F32, 8,
                     scratch.data_ptr(), sb, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(y[:17], few), M
        ref = xm.float() @ w.float().T
        torch.testing.assert_close(y, base[:M] + ref, rtol=1e-4, atol=1e-4 * ref.abs().max().item())
        assert int(scratch[:4].view(torch.int32).item()) == 0


@pytest.mark.parametrize("M,split", [(3, 1), (100, 1), (100, 8), (300, 4)])
@pytest.mark.parametrize("shift", [1, 2])
def test_linear_takes_a_scratch_at_any_address(gs, M, split, shift):
    """The scratch has no alignment rule: launches that do not sum partials in it
    only clear it, and the same bytes come out at any address."""
    N, K = 1024, 4096
    g = torch.Generator(device=DEV).manual_seed(M + split)
    x = torch.randn(M, K, device=DEV, generator=g).half()
    w = (0.02 * torch.randn(N, K, device=DEV, generator=g)).half()
    want = torch.zeros(M, N, dtype=torch.float16, device=DEV)
    _linear(gs, x, w, M, N, K, gs.EPI_STORE_F16, split, want)
    y = torch.zeros_like(want)
    sb = gs.gs_linear_scratch_bytes(M, N, split)
    scratch = torch.full((sb + 4,), 0x7F, dtype=torch.uint8, device=DEV)
    gs.gs_linear(x.data_ptr(), w.data_ptr(), y.data_ptr(), M, N, K, gs.EPI_STORE_F16, split,
                 scratch.data_ptr() + shift, sb, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    assert not scratch[shift:shift + 4].any() and int(scratch[0]) == 0x7F


@pytest.mark.parametrize("epi,N", [(0, 1024), (2, 1024), (3, 2048)])
def test_clusters_above_64_rows_other_epilogues(gs, epi, N):
    """fp16 stores, SwiGLU and argmax keys of 100 rows in clusters of eight (at most
    256 CTAs): every row has the bits it has alone in a window of its own 17."""
    M, K = 100, 4096
    g = torch.Generator(device=DEV).manual_seed(epi)
    x = torch.randn(M, K, device=DEV, generator=g).half()
    w = (0.02 * torch.randn(2 * N if epi == gs.EPI_SWIGLU else N, K, device=DEV, generator=g)).half()

    def out(m):
        return (torch.zeros(m, dtype=torch.int64, device=DEV) if epi == gs.EPI_ARGMAX
                else torch.zeros(m, N, dtype=torch.float16, device=DEV))

    y = out(M)
    _linear(gs, x, w, M, N, K, epi, 8, y)
    for m0 in range(0, M, 17):
        m = min(17, M - m0)
        part = out(m)
        _linear(gs, x[m0:m0 + m].contiguous(), w, m, N, K, epi, 8, part)
        assert torch.equal(y[m0:m0 + m], part), m0


@pytest.mark.parametrize("items", [9, 16, 17, 32, 33, 54])
@pytest.mark.parametrize("W,Hq,Hkv", [(5, 16, 8), (16, 16, 2)])
def test_attention_merges_many_items(gs, items, W, Hq, Hkv):
    """One-page items beyond eight, up to the interface's 54, merged through global
    scratch: their maxima and sums are read sixteen at a time (blocks of 10 and of
    128 rows)."""
    B = 40 if Hkv == 2 else 6                  # more than one wave of CTAs
    rng = np.random.default_rng(items)
    ns = [64 * items - 40] + [int(v) for v in rng.integers(1, 64 * items - 40, B - 1)]
    q, k, v = synth.attn_inputs(B, W, 64 * items, Hq, Hkv, index=items)
    pool, pt, _ = _paged(k, v, rng)
    got = _run_attention(gs, 1, q, pool, pt, np.array(ns), W, Hq, Hkv, 1)
    for b in (0, 1, int(np.argmin(ns))):
        allowed = od.verify_allowed(ns[b], W - 1)
        nk = allowed.shape[1]
        want = _oracle_attn(q[b].astype(np.float64), k[b, :nk].astype(np.float64),
                            v[b, :nk].astype(np.float64), allowed, Hq, Hkv)
        np.testing.assert_allclose(got[b], want, rtol=5e-3, atol=5e-3)


@pytest.mark.parametrize("N,K,split", [(256, 640, 5), (512, 1216, 19), (384, 2048, 32)])
@pytest.mark.parametrize("epi", [0, 1, 3])
def test_split_sums_through_scratch(gs, N, K, split, epi):
    """Splits that form no cluster, around the slices of 8 and 32 tokens in which the
    last CTA adds them up, with the splits' remainders: a row's bits are those of the
    64-row window, and the allocation-free call's tiles of up to 256 rows give the
    same."""
    g = torch.Generator(device=DEV).manual_seed(N + split)
    x = torch.randn(137, K, device=DEV, generator=g).half()
    w = (0.05 * torch.randn(N, K, device=DEV, generator=g)).half()
    base = torch.randn(137, N, device=DEV, generator=g)

    def out(m):
        if epi == gs.EPI_RESID_F32:
            return base[:m].clone()
        return (torch.zeros(m, dtype=torch.int64, device=DEV) if epi == gs.EPI_ARGMAX
                else torch.zeros(m, N, dtype=torch.float16, device=DEV))

    want = out(137)
    _linear(gs, x, w, 137, N, K, epi, split, want)     # chunks inside each CTA
    for M in (1, 7, 8, 9, 32, 33, 40, 41, 64):
        y = out(M)
        _linear(gs, x[:M].contiguous(), w, M, N, K, epi, split, y)
        assert torch.equal(y, want[:M]), M
    stream = torch.cuda.current_stream().cuda_stream
    for M in (8, 9, 72, 73) + ((136, 137) if split == 5 else ()):   # (partials within 8 MiB)
        xm, y = x[:M].contiguous(), out(M)
        gs.gs_linear_noalloc(xm.data_ptr(), w.data_ptr(), y.data_ptr(), M, N, K, epi, split, stream)
        assert gs.gs_linear_noalloc_status(stream) == gs.GS_OK
        assert torch.equal(y, want[:M]), M


@pytest.mark.parametrize("tiles,K,Ms", [
    (153, 256, (1, 32, 33, 64, 65, 128, 129)), (228, 192, (17, 64, 100, 128)), (229, 192, (17, 64, 128)),
    (160, 8192, (40, 192, 193, 256, 257)),
])
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
def test_one_to_two_tiles_per_sm(gs, tiles, K, Ms, epi):
    """Unsplit launches of a little more than one wave, on both sides of the sizes up
    to which they take a CTA per tile: a row's bits are those of the 300-row window
    (the persistent kernel), and the fp32 matmul is near."""
    N = tiles * 64 if epi == gs.EPI_SWIGLU else tiles * 128
    g = torch.Generator(device=DEV).manual_seed(tiles + epi)
    x = torch.randn(300, K, device=DEV, generator=g).half()
    w = (0.02 * torch.randn(tiles * 128, K, device=DEV, generator=g)).half()
    base = torch.randn(300, N, device=DEV, generator=g)

    def out(m):
        if epi == gs.EPI_RESID_F32:
            return base[:m].clone()
        return (torch.zeros(m, dtype=torch.int64, device=DEV) if epi == gs.EPI_ARGMAX
                else torch.zeros(m, N, dtype=torch.float16, device=DEV))

    want = out(300)
    _linear(gs, x, w, 300, N, K, epi, 1, want)
    for M in Ms:
        y = out(M)
        _linear(gs, x[:M].contiguous(), w, M, N, K, epi, 1, y)
        assert torch.equal(y, want[:M]), M
    if epi == gs.EPI_STORE_F16:
        ref = x.float() @ w.float().T
        torch.testing.assert_close(want.float(), ref, rtol=2e-3, atol=1e-3 * ref.abs().max().item())
