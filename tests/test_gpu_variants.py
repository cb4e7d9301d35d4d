"""GPU side of the variants around the path: 16-bit metadata (Section 3.2), the decoder's optional
renormalisation (Section A.3), the alpha grid (Section B.2) and the on-disk blob."""
import ctypes as C
import os

import numpy as np
import pytest
import torch

from conftest import load_golden_codebook

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2605_26339_b200 import binding as q
    from paper_2605_26339_b200 import blob
    from paper_2605_26339_b200.model_codec import choose_alpha

DEV = "cuda:0"


def _bits(t):
    return t.cpu().view(torch.int16).numpy().view(np.uint16)


def _encode(W, act, alpha, block, K, round16=False):
    d_out, d_in = W.shape
    cbh = load_golden_codebook(K)
    cb = q.Codebook(cbh)
    s = torch.from_numpy(q.channel_scales(act, alpha)).to(DEV)
    signs = torch.from_numpy(q.make_signs(q.DEFAULT_SIGN_SEED, d_in)).to(DEV)
    Wd = W.to(DEV)
    p = q.make_params(Wd, d_out, d_in, block, K, 0, (q.packed_row_bytes(d_in, K) + 15) // 16 * 16)
    if round16:
        q.round_f16(s)
    sigma = torch.empty(d_in // 2, dtype=torch.float32, device=DEV)
    ws = torch.empty(q.calibrate_workspace_bytes(p), dtype=torch.uint8, device=DEV)
    q.calibrate(Wd, p, s, signs, sigma, ws)
    if round16:
        q.round_f16(sigma)
    packed = torch.empty((d_out, p.packed_row_stride), dtype=torch.uint8, device=DEV)
    norm = torch.empty(d_out, dtype=torch.float32, device=DEV)
    q.encode(Wd, p, s, signs, sigma, cb, packed, norm)
    if round16:
        q.round_f16(norm)
    return dict(cb=cb, cbh=cbh, s=s, signs=signs, W=Wd, p=p, sigma=sigma, packed=packed, norm=norm)


def _problem(seed, d_out=96, d_in=2048):
    g = torch.Generator().manual_seed(seed)
    W = (torch.randn((d_out, d_in), generator=g) * torch.exp(0.7 * torch.randn((d_out, 1), generator=g))).to(torch.bfloat16)
    act = torch.exp(torch.randn(d_in, generator=g)).numpy().astype(np.float32)
    return W, act


def test_round_f16_matches_oracle(orc):
    rng = np.random.default_rng(4)
    v = (rng.standard_normal(100003) * np.exp(rng.uniform(-22, 13, 100003))).astype(np.float32)
    v[:6] = [0.0, 65504.0, 65520.0, 2.0 ** -24, 2.0 ** -25, -1e9]
    t = torch.from_numpy(v.copy()).to(DEV)
    q.round_f16(t)
    assert np.array_equal(t.cpu().numpy(), orc.round_f16(v))


def test_renormalised_decode(orc):
    W, act = _problem(31)
    e = _encode(W, act, 0.3, 128, 256)
    adj = torch.empty_like(e["norm"])
    q.renorm_row_norms(e["packed"], e["norm"], e["sigma"], e["cb"], e["p"], adj)
    ref = orc.renorm_row_norms(e["packed"].cpu().numpy(), e["norm"].cpu().numpy(), e["sigma"].cpu().numpy(), e["cbh"], 2048)
    np.testing.assert_allclose(adj.cpu().numpy(), ref, rtol=2e-7)
    # decoding with the factors restores the stored norm of the scaled row
    what = torch.empty(W.shape, dtype=torch.bfloat16, device=DEV)
    q.decode(e["packed"], adj, e["s"], e["signs"], e["sigma"], e["cb"], e["p"], what)
    length = ((what.float() * e["s"]) ** 2).sum(1).sqrt()
    assert torch.allclose(length, e["norm"], rtol=2e-3)  # bf16 rounding of 2048 outputs
    q.decode(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], e["p"], what)
    plain = ((what.float() * e["s"]) ** 2).sum(1).sqrt()
    assert torch.allclose(plain, e["norm"] * e["norm"] / adj, rtol=2e-3)  # the plain decoder's length is r |yhat|
    assert not torch.allclose(plain, e["norm"], rtol=1e-4)


def test_f16_metadata_round_trip_through_a_blob(orc, tmp_path):
    """16-bit metadata end to end: scales and sigma rounded before encoding, norms after; the blob on
    disk (f16 metadata) decodes on the GPU to the very bits the in-memory arrays decode to, and the
    radial error added by the rounded norms stays within half an f16 ulp (2^-11 relative)."""
    W, act = _problem(32)
    e = _encode(W, act, 0.3, 128, 2048, round16=True)
    exact = _encode(W, act, 0.3, 128, 2048, round16=False)
    rel = (e["norm"] - exact["norm"]).abs() / exact["norm"]
    assert float(rel.max()) <= 2.0 ** -11 * 1.01 + 1e-3  # sigma / scales differ slightly too (<= 1e-3 on r)
    what = torch.empty(W.shape, dtype=torch.bfloat16, device=DEV)
    q.decode(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], e["p"], what)
    path = os.path.join(tmp_path, "m.qamw")
    size = blob.save_blob(path, d_out=96, d_in=2048, block=128, K=2048, alpha=0.3, sign_seed=q.DEFAULT_SIGN_SEED,
                          codebook=e["cbh"], sigma=e["sigma"].cpu().numpy(), row_norm=e["norm"].cpu().numpy(),
                          packed=e["packed"].cpu().numpy(), chan_scale=e["s"].cpu().numpy(), f16_metadata=True)
    b = blob.load_blob(path)
    cb2 = q.Codebook(b["codebook"])
    p2 = q.make_params(None, b["d_out"], b["d_in"], b["block"], b["K"], 0, b["packed_row_stride"])
    signs2 = torch.from_numpy(q.make_signs(b["sign_seed"], b["d_in"])).to(DEV)
    what2 = torch.empty(W.shape, dtype=torch.bfloat16, device=DEV)
    q.decode(torch.from_numpy(b["packed"]).to(DEV), torch.from_numpy(b["row_norm"]).to(DEV),
             torch.from_numpy(b["chan_scale"]).to(DEV), signs2, torch.from_numpy(b["sigma"]).to(DEV), cb2, p2, what2)
    assert np.array_equal(_bits(what), _bits(what2))
    # against the oracle on the same rounded metadata
    ref = orc.decode(b["packed"], b["row_norm"], 128, b["codebook"], b["chan_scale"], signs2.cpu().numpy(), b["sigma"], 2048)
    d = np.abs(_bits(what2).astype(np.int32) - ref.astype(np.int32))
    assert (d <= 1).mean() > 0.9998
    assert size < 96 * 2048 * 6 / 8 + 2048 * 8 + 8192  # about 5.5 bits per weight plus the codebook


def test_alpha_grid_picks_the_lowest_output_error(orc):
    W, act = _problem(33, 64, 1024)
    act[::50] *= 30.0  # a few loud channels make the scaling matter
    cb = q.Codebook(load_golden_codebook(256))
    best, scores = choose_alpha(W.to(DEV), torch.from_numpy(act).to(DEV), cb, 128)
    assert set(scores) == {0.0, 0.3, 0.5, 0.8} and best == min(scores, key=lambda a: scores[a][1])
    assert scores[best][1] < scores[0.0][1]  # scaling helps the activation-weighted error here
    # one grid point against the oracle's round trip
    s = orc.channel_scales(act, float(np.float32(0.5)))
    signs = orc.make_signs(q.DEFAULT_SIGN_SEED, 1024)
    Wb = _bits(W)
    sigma, _ = orc.calibrate(Wb, 128, s, signs)
    enc = orc.encode(Wb, 128, cb.host, s, signs, sigma)
    what = orc.decode(enc["packed"], enc["row_norm"], 128, cb.host, s, signs, sigma, 1024)
    d = orc.distortion(Wb, what, act)
    assert abs(np.sqrt(d[2] / d[3]) - scores[0.5][1]) < 2e-3 * scores[0.5][1]


@pytest.mark.parametrize("d_out,d_in,block,K,n_vec", [(300, 2048, 128, 2048, 1), (129, 5120, 128, 256, 4),
                                                      (64, 13824, 256, 2048, 2), (40, 1024, 32, 128, 1),
                                                      (33, 512, 1024 // 2, 4096, 1), (1000, 2048, 1024, 2048, 4),
                                                      (7, 64, 2, 64, 2), (50, 11008, 64, 1024, 1)])
def test_fused_decode_gemv(orc, d_out, d_in, block, K, n_vec):
    """y = W_hat x from the packed stream against the oracle's decoder (f64, before the bf16 rounding)
    followed by a plain matrix product.  The kernel accumulates in f32: the error of a row stays below
    1e-5 |w_hat_i| |x| (d_in terms, each product and sum rounded to 2^-24 relative)."""
    W, act = _problem(50 + n_vec, d_out, d_in)
    e = _encode(W, act, 0.3, block, K)
    g = torch.Generator().manual_seed(d_in)
    x = torch.randn((n_vec, d_in), generator=g)
    y = torch.full((d_out, n_vec), float("nan"), dtype=torch.float32, device=DEV)
    q.decode_gemv(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], e["p"], x.to(DEV), y)
    # the layout-agnostic kernel (taken for packed rows that are not 16-byte aligned) gives the same product
    y_general = torch.full_like(y, float("nan"))
    pg = q.make_params(None, d_out, d_in, block, K, q.FLAG_GENERAL_KERNELS, e["p"].packed_row_stride)
    q.decode_gemv(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], pg, x.to(DEV), y_general)
    _, w64 = orc.decode(e["packed"].cpu().numpy(), e["norm"].cpu().numpy(), block, e["cbh"], e["s"].cpu().numpy(),
                        e["signs"].cpu().numpy(), e["sigma"].cpu().numpy(), d_in, want_f64=True)
    ref = w64 @ x.numpy().astype(np.float64).T
    bound = 1e-5 * np.sqrt((w64 ** 2).sum(1))[:, None] * np.sqrt((x.numpy().astype(np.float64) ** 2).sum(1))[None, :]
    assert np.all(np.abs(y.cpu().numpy() - ref) <= bound + 1e-30)
    assert np.all(np.abs(y_general.cpu().numpy() - ref) <= bound + 1e-30)
    # and against the two-step pipeline of the paper (decode to bf16, then multiply): bf16 rounding only
    what = torch.empty((d_out, d_in), dtype=torch.bfloat16, device=DEV)
    q.decode(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], e["p"], what)
    two_step = what.double() @ x.to(DEV).double().T
    assert torch.allclose(y.double(), two_step, rtol=0, atol=float(2.0 ** -7 * np.abs(ref).max() + 1e-30))


def test_fused_gemv_argument_errors():
    lv = load_golden_codebook(64)
    cb = q.Codebook(lv)
    dummy = torch.zeros(4096, dtype=torch.uint8, device=DEV)
    f = torch.zeros(4096, dtype=torch.float32, device=DEV)
    p = q.make_params(None, 4, 48, 16, 64)  # d_in not a multiple of 32
    with pytest.raises(q.QamwError) as e:
        q.decode_gemv(dummy, f, None, dummy, f, cb, p, f[:48].reshape(1, 48), f[:4].reshape(4, 1), dummy)
    assert e.value.code == q.ERR_SHAPE
    p = q.make_params(None, 4, 64, 16, 64)
    with pytest.raises(q.QamwError) as e:
        q.decode_gemv(dummy, f, None, dummy, f, cb, p, f[:192].reshape(3, 64), f[:12].reshape(4, 3), dummy)  # 3 vectors
    assert e.value.code == q.ERR_ARG


def test_step_replayed_as_a_cuda_graph_gives_the_same_bytes():
    """The batched step captured into one CUDA graph: replaying it reproduces the packed stream, the row
    norms, the decoded matrices and the distortion sums of the eager step bit for bit."""
    from paper_2605_26339_b200 import synth
    from paper_2605_26339_b200.model_codec import ModelCodec
    spec = synth.workload("cfg2", 256)
    mc = ModelCodec.from_synthetic(spec, torch.device(DEV), load_golden_codebook(256), layers=[0])
    mc.step()
    torch.cuda.synchronize()
    want = [(s.packed.clone(), s.row_norm.clone(), s.w_hat.clone(), s.dist.clone()) for s in mc.slots]
    graph = mc.capture_step()
    for s in mc.slots:
        s.packed.zero_(); s.row_norm.zero_(); s.w_hat.zero_(); s.dist.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for s, (p, r, w, d) in zip(mc.slots, want):
        assert torch.equal(s.packed, p) and torch.equal(s.row_norm, r)
        assert torch.equal(s.w_hat.view(torch.int16), w.view(torch.int16)) and torch.equal(s.dist, d)
    assert int(mc.status.cpu()[0]) == 0


@pytest.mark.parametrize("K", [2, 32, 64, 128, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("d_out,d_in,n_vec", [(1, 32, 1), (150, 544, 2), (301, 1056, 1), (37, 2080, 4)])
def test_fused_gemv_rows_off_16_byte_boundaries(orc, K, d_out, d_in, n_vec):
    """Every index width, with packed rows that start anywhere on 4 bytes and end inside a 16-byte piece."""
    W, act = _problem(K + n_vec, d_out, d_in)
    g = torch.Generator().manual_seed(d_in)
    cbh = orc.train_codebook(K, 1 << 13, 7, 2, 1e-6)[0]
    cb = q.Codebook(cbh)
    p = q.make_params(None, d_out, d_in, 32, K)
    packed = torch.randint(0, 256, (d_out, p.packed_row_stride), generator=g, dtype=torch.uint8)
    norm, sigma = torch.rand(d_out, generator=g) + 0.5, torch.rand(d_in // 2, generator=g) + 0.5
    s = torch.from_numpy(q.channel_scales(act, 0.3))
    signs = torch.from_numpy(q.make_signs(q.DEFAULT_SIGN_SEED, d_in))
    x = torch.randn((n_vec, d_in), generator=g)
    y = torch.full((d_out, n_vec), float("nan"), dtype=torch.float32, device=DEV)
    q.decode_gemv(packed.to(DEV), norm.to(DEV), s.to(DEV), signs.to(DEV), sigma.to(DEV), cb, p, x.to(DEV), y)
    _, w64 = orc.decode(packed.numpy(), norm.numpy(), 32, cbh, s.numpy(), signs.numpy(), sigma.numpy(), d_in, want_f64=True)
    ref = w64 @ x.numpy().astype(np.float64).T
    bound = 1e-5 * np.sqrt((w64 ** 2).sum(1))[:, None] * np.sqrt((x.numpy().astype(np.float64) ** 2).sum(1))[None, :]
    assert np.all(np.abs(y.cpu().numpy() - ref) <= bound + 1e-30)


@pytest.mark.parametrize("d_in", [2, 1024, 1026, 2050, 4098, 8064, 8066, 16384])
@pytest.mark.parametrize("alpha", [0.0, 0.3])
def test_quantize_prepares_the_columns_as_the_host_functions_do(d_in, alpha):
    """Channel scales and signs that qamw_quantize computes on the device, around every size of its parameter blocks."""
    W, act = _problem(d_in, 3, d_in)
    act[0], act[-1] = 0.0, 1e30
    cb = q.Codebook(load_golden_codebook(64))
    Wd = W.to(DEV)
    p = q.make_params(Wd, 3, d_in, 2, 64)
    new = lambda n, dt: torch.empty(n, dtype=dt, device=DEV)
    s, signs, sigma, norm = new(d_in, torch.float32), new(d_in, torch.int8), new(d_in // 2, torch.float32), new(3, torch.float32)
    packed, ws = new((3, p.packed_row_stride), torch.uint8), new(max(8, q.calibrate_workspace_bytes(p)), torch.uint8)
    host = act.copy()
    q.quantize(Wd, p, host, alpha, 123456789, cb, s, signs, sigma, packed, norm, ws)
    host[:] = -1.0  # the statistics belong to the caller again
    assert np.array_equal(signs.cpu().numpy(), q.make_signs(123456789, d_in))
    if alpha:
        np.testing.assert_allclose(s.cpu().numpy(), q.channel_scales(act, alpha), rtol=1.2e-7)


def test_a_refused_launch_is_reported_once():
    """A launch that the runtime refuses on the host is the error of the call that made it, and of no later one.  The
    refusal: work for the default stream while another stream that synchronises with it is being captured."""
    rt = C.CDLL("libcudart.so.12")  # torch's copy, loaded already
    W, act = _problem(51, 8, 256)
    W = W.to(DEV)
    p = q.make_params(W, 8, 256, 64, 256)
    signs = torch.from_numpy(q.make_signs(1, 256)).to(DEV)
    y, norm = torch.empty((8, 256), device=DEV), torch.empty(8, device=DEV)
    half = torch.ones(4, device=DEV)
    q.rotate(W, p, None, signs, y, norm)
    torch.cuda.synchronize()
    stream, graph = C.c_void_p(), C.c_void_p()
    assert rt.cudaStreamCreate(C.byref(stream)) == 0
    try:
        assert rt.cudaStreamBeginCapture(stream, 0) == 0
        try:
            with pytest.raises(q.QamwError) as e:
                q.rotate(W, p, None, signs, y, norm)
            assert e.value.code == q.ERR_CUDA
        finally:
            rt.cudaStreamEndCapture(stream, C.byref(graph))  # the refusal has ended the capture
            rt.cudaGetLastError()
        q.round_f16(half)
        out = q.train_codebook_gpu(2, 4096, 0, 2)
        assert out["iters"] == 2 and np.isfinite(out["codebook"]).all()
    finally:
        assert rt.cudaStreamDestroy(stream) == 0


def test_outputs_that_share_memory_until_they_are_written(orc):
    """An output tensor that still shares its memory with another (a lazy clone) takes its own before the call writes."""
    W, act = _problem(52, 16, 256)
    e = _encode(W, act, 0.3, 64, 256)
    plain = torch.empty((16, 256), dtype=torch.bfloat16, device=DEV)
    q.decode(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], e["p"], plain)
    base = torch.zeros_like(plain)
    out = torch._lazy_clone(base)
    q.decode(e["packed"], e["norm"], e["s"], e["signs"], e["sigma"], e["cb"], e["p"], out)
    assert torch.equal(out, plain) and not base.any()
    packed, norm = torch.zeros_like(e["packed"]), torch.zeros_like(e["norm"])
    q.encode(e["W"], e["p"], e["s"], e["signs"], e["sigma"], e["cb"], torch._lazy_clone(packed), torch._lazy_clone(norm))
    assert not packed.any() and not norm.any()


def test_quotients_of_the_column_factors(tmp_path):
    """quotient2 equals the correctly rounded division for every significand of the divisor, at both ends of the range that it is
    used for and in its middle, and for the numerator of every block size."""
    import os
    import subprocess
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src = tmp_path / "quotient.cu"
    src.write_text(r'''
#include <cmath>
#include <cstdio>
#include "qamw_device.cuh"
__global__ void check(float a, int exponent, unsigned long long* wrong) {
    const unsigned m = 2u * (blockIdx.x * blockDim.x + threadIdx.x);  // 2^23 significands, two at a time
    const float b0 = __uint_as_float((unsigned(exponent + 127) << 23) | m), b1 = __uint_as_float((unsigned(exponent + 127) << 23) | (m + 1u));
    float q0, q1;
    unpack2(quotient2(pack2(a, a), b0, b1), q0, q1);
    if (q0 != __fdiv_rn(a, b0) || q1 != __fdiv_rn(a, b1)) atomicAdd(wrong, 1ull);
}
int main() {
    unsigned long long* wrong;
    if (cudaMallocManaged(&wrong, 8) != cudaSuccess) return 1;
    *wrong = 0;
    for (int log2b = 1; log2b <= 10; ++log2b)
        for (int e : {-60, -5, -1, 0, 1, 4, 59}) check<<<(1 << 22) / 256, 256>>>(float(1.0 / std::sqrt(double(1 << log2b))), e, wrong);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    std::printf("%llu", *wrong);
}
''')
    exe = tmp_path / "quotient"
    from paper_2605_26339_b200 import build
    subprocess.run([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-I",
                    os.path.join(root, "paper_2605_26339_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "0"


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -61, 2.0 ** 61])
def test_decode_with_channel_scales_off_the_usual_range(scale):
    """Channel scales below and above the range of quotient2, alone and among usual ones: as the general kernels, bit for bit."""
    d_out, d_in, K = 37, 1056, 64
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    cb = q.Codebook(q.train_codebook(K, n_samples=4096, seed=1, max_iters=3)[0])
    s = torch.rand(d_in, generator=g, device=DEV) + 0.5
    s[::7] *= scale
    signs = torch.from_numpy(q.make_signs(q.DEFAULT_SIGN_SEED, d_in)).to(DEV)
    sigma = torch.rand(d_in // 2, generator=g, device=DEV) + 0.1
    p = q.make_params(torch.empty((d_out, d_in), dtype=torch.bfloat16, device=DEV), d_out, d_in, 32, K)
    packed = torch.randint(0, 256, (d_out, p.packed_row_stride), generator=g, device=DEV, dtype=torch.uint8)
    norm = torch.rand(d_out, generator=g, device=DEV)
    out = [torch.empty((d_out, d_in), dtype=torch.bfloat16, device=DEV) for _ in range(2)]
    for o, flags in zip(out, (0, q.FLAG_GENERAL_KERNELS)):
        p.flags = flags
        q.decode(packed, norm, s, signs, sigma, cb, p, o)
    assert torch.equal(out[0].view(torch.int16), out[1].view(torch.int16))


@pytest.mark.parametrize("kind", ["ordinary", "subnormal", "huge", "inf", "nan", "inf and huge"])
@pytest.mark.parametrize("batched", [False, True])
def test_distortion_of_numbers_at_the_ends_of_the_range(kind, batched):
    """The four sums against doubles for reconstructions with subnormal, huge and non-finite entries, also beside weights as large."""
    d_out, d_in = 37, 1048
    g = torch.Generator(device=DEV)
    g.manual_seed(4)
    W = torch.randn((d_out, d_in), generator=g, device=DEV).to(torch.bfloat16)
    h = (W.float() * (1 + 0.1 * torch.randn((d_out, d_in), generator=g, device=DEV))).to(torch.bfloat16)
    act = torch.rand(d_in, generator=g, device=DEV) + 0.5
    big = 3.3895313892515355e38  # the largest bf16
    if kind == "subnormal":
        W, h = (W.float() * 2.0 ** -130).to(torch.bfloat16), (h.float() * 2.0 ** -130).to(torch.bfloat16)
        assert (h != 0).any() and h.float().abs().max() < 2.0 ** -126
    elif kind == "huge":
        W[5, 7], h[5, 7], h[20, 100], W[36, 1047] = big, -big, big, -big
    elif kind == "inf":
        h[3, 9], h[30, 1040] = float("inf"), -float("inf")
    elif kind == "nan":
        h[17, 511] = float("nan")
    elif kind == "inf and huge":
        W[3, 9], h[3, 9] = big, float("inf")
    p = q.make_params(W, d_out, d_in, 8, 64)
    out = torch.zeros(4, dtype=torch.float64, device=DEV)
    if batched:
        cb = q.Codebook(q.train_codebook(64, n_samples=4096, seed=1, max_iters=3)[0])
        signs = torch.from_numpy(q.make_signs(q.DEFAULT_SIGN_SEED, d_in)).to(DEV)
        sigma = torch.ones(d_in // 2, device=DEV)
        packed = torch.zeros((d_out, p.packed_row_stride), dtype=torch.uint8, device=DEV)
        norm = torch.ones(d_out, device=DEV)
        q.Batch([q.make_matrix(p, W, None, signs, sigma, act, packed, norm, h, out)], cb).distortion()
    else:
        q.distortion(W, h, act, p, out)
    w, r2 = W.double(), act.double() ** 2
    e2 = (w - h.double()) ** 2
    want = torch.stack([e2.sum(), (w * w).sum(), (r2 * e2).sum(), (r2 * w * w).sum()])
    assert torch.allclose(out, want, rtol=1e-12, atol=0.0, equal_nan=True), (out, want)
