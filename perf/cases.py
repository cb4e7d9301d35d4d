"""The calls that a user of the codec makes, at the sizes and options they are made with.

Five kinds of call, each through the package's public entry points:
  quantize  one matrix in one call: channel scales, signs, pair scales, packed stream and row norms
  model     all matrices of one or more decoder layers behind one handle: calibrate, encode, decode, distortion
  decode    one matrix back to bf16
  gemv      the product of a packed matrix with 1, 2 or 4 activation vectors
  train     a codebook fitted to given pairs on the device

Weights and activation statistics follow `synth`: heavy-tailed or normal entries, a scale per row, outlier
channels.  Codebooks are trained once per size, as a program keeps one per bitrate.
"""
import functools
import math

import numpy as np
import torch

from paper_2605_26339_b200 import binding as q
from paper_2605_26339_b200 import model_codec, synth

DEV = "cuda"
ALPHA = 0.3
MAX_WEIGHTS = {"quantize": 13824 * 5120, "model": 4 * synth.workload("cfg3").n_weights // 40, "decode": 13824 * 5120,
               "gemv": 13824 * 5120}


def _matrix(name, kind, d_out, d_in, block, K, dtype="bf16", entry="student_t", **more):
    return dict(name=name, kind=kind, d_out=d_out, d_in=d_in, block=block, K=K, dtype=dtype, entry=entry, **more)


def _layers(name, hidden, inter, kv, layers, block, K, dtype="bf16", entry="student_t"):
    return dict(name=name, kind="model", hidden=hidden, inter=inter, kv=kv, layers=layers, block=block, K=K, dtype=dtype,
                entry=entry)


def listed():
    return [
        # a single small f32 layer (benchmark configuration 0): launches and host work count
        _matrix("quantize f32 1024x1024", "quantize", 1024, 1024, 128, 256, "f32", "normal"),
        # an attention projection of a 7B model with the block size that the paper's rule gives for it
        _matrix("quantize 4096x4096 b1024", "quantize", 4096, 4096, 1024, 2048),
        # a width that is no multiple of 16 (small Hadamard blocks) and an odd number of rows
        _matrix("quantize ragged 1013x1000", "quantize", 1013, 1000, 8, 256, "bf16", "normal"),
        # one layer of a 1.1B model (configuration 2): seven small matrices, some with 256 rows
        _layers("layer 1.1B", 2048, 5632, 256, 1, 128, 2048, "bf16", "normal"),
        # one layer of a 7B model (configuration 1)
        _layers("layer 7B", 4096, 11008, 4096, 1, 128, 2048),
        # four layers of a 13B model (a piece of configuration 3): the bulk of quantising a checkpoint
        _layers("4 layers 13B", 5120, 13824, 5120, 4, 128, 2048),
        # the smallest matrix of a 1.1B model, expanded before its product
        _matrix("decode 256x2048", "decode", 256, 2048, 128, 2048, "bf16", "normal"),
        # the largest matrix of a 13B model (configuration 4)
        _matrix("decode 13824x5120", "decode", 13824, 5120, 128, 2048),
        # rows whose packed length is no multiple of 16 bytes
        _matrix("decode ragged 2999x2744", "decode", 2999, 2744, 8, 512),
        # token by token generation from the packed weights: 1.1B model, one sequence
        _matrix("gemv 2048x5632 x1", "gemv", 2048, 5632, 128, 2048, "bf16", "normal", n_vec=1),
        # the same for a 13B model, four sequences at once
        _matrix("gemv 13824x5120 x4", "gemv", 13824, 5120, 128, 2048, n_vec=4),
        # a codebook of the default size fitted to a checkpoint's own pairs, default number of pairs and limits
        dict(name="train K2048", kind="train", K=2048, n=1 << 20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rule(d_in):
    return min(1024, d_in & -d_in)


def draw(rng):
    kind = rng.choice(["quantize", "quantize", "model", "model", "decode", "decode", "gemv", "gemv", "train"])
    K = 1 << rng.choice([6, 7, 8, 9, 10, 11, 11, 11, 12])
    if kind == "train":
        K = min(K, 2048)
        return dict(kind=kind, K=K, n=_log(rng, 1 << 16, 1 << 20))
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    entry = rng.choice(["student_t", "normal"])
    if kind == "model":
        hidden = 128 * _log(rng, 8, 40)
        inter = 128 * min(108, int(hidden / 128 * rng.uniform(2.0, 3.5)))
        kv = rng.choice([hidden, 128 * rng.randint(1, 8)])
        one = 2 * hidden * (hidden + kv) + 3 * hidden * inter
        layers = rng.randint(1, max(1, min(4, MAX_WEIGHTS[kind] // (one * (2 if dtype == "f32" else 1)))))
        return dict(kind=kind, hidden=hidden, inter=inter, kv=kv, layers=layers, block=rng.choice([64, 128, 128]), K=K,
                    dtype=dtype, entry=entry)
    d_in = 64 * _log(rng, 8, 216)
    if kind != "gemv" and rng.random() < 0.3:
        d_in = 8 * _log(rng, 64, 1000) + 8  # often no multiple of 16
    d_out = _log(rng, 256, min(13824, MAX_WEIGHTS[kind] // (d_in * (2 if dtype == "f32" else 1))))
    case = dict(kind=kind, d_out=d_out, d_in=d_in, block=min(_rule(d_in), rng.choice([64, 128, 128, 256, 1024])), K=K,
                dtype=dtype, entry=entry)
    if kind == "gemv":
        case["n_vec"] = rng.choice([1, 1, 2, 4])
    return case


# ------------------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _codebook(K):
    """The codebook handle of one bitrate, kept for the life of the program."""
    return q.Codebook(q.train_codebook(K, n_samples=max(1 << 15, 16 * K), seed=K, max_iters=12)[0])


def _spec(case, matrices, layers):
    heavy = case["entry"] == "student_t"
    return synth.WorkloadSpec("case", tuple(matrices), layers, case["dtype"], case["entry"], 4 if heavy else 0,
                              0.7 if heavy else 0.5, 0.01 if heavy else 0.0, 20.0, 0.01, 20.0, ALPHA, case["block"], case["K"], 0)


def _quantize(s):
    q.quantize(s["W"], s["p"], s["act"], ALPHA, q.DEFAULT_SIGN_SEED, s["cb"], s["scale"], s["signs"], s["sigma"], s["packed"],
               s["norm"], s["ws"], s["status"])


def _one(case, seed):
    """One weight matrix with everything that quantising it needs, outputs allocated."""
    d_out, d_in, K = case["d_out"], case["d_in"], case["K"]
    m = synth.MatrixSpec("w", d_out, d_in)
    spec = _spec(case, [m], 1)
    W = synth.make_weight(spec, m, seed, device=DEV)
    act = synth.make_act_rms(spec, d_in, seed, device=DEV).cpu().numpy()
    p = q.make_params(W, d_out, d_in, case["block"], K)
    new = functools.partial(torch.empty, device=DEV)
    return dict(W=W, act=act, p=p, cb=_codebook(K), scale=new(d_in), signs=new(d_in, dtype=torch.int8), sigma=new(d_in // 2),
                packed=new((d_out, p.packed_row_stride), dtype=torch.uint8), norm=new(d_out),
                ws=new(max(8, q.calibrate_workspace_bytes(p)), dtype=torch.uint8),
                status=torch.zeros(1, dtype=torch.int32, device=DEV))


class _Arena:
    """One buffer cut into pieces that start on 256 bytes; what lies between them stays zero."""

    def __init__(self, dtype, counts):
        self.item = torch.empty(0, dtype=dtype).element_size()
        self.size = [-(-n * self.item // 256) * 256 // self.item for n in counts]
        self.all = torch.zeros(sum(self.size), dtype=dtype, device=DEV)
        self.at = 0

    def take(self, i, shape):
        v = self.all[self.at:self.at + math.prod(shape)].view(shape)
        self.at += self.size[i]
        return v


def _model(case, seed):
    """All matrices of the layers behind one ModelCodec; outputs of one kind share a buffer."""
    spec = _spec(case, synth.decoder_layer(case["hidden"], case["inter"], case["kv"]), case["layers"])
    mats = list(synth.iter_matrices(spec))
    K, stride = case["K"], lambda m: q.default_packed_row_stride(m.d_in, case["K"])
    out = dict(packed=_Arena(torch.uint8, [m.d_out * stride(m) for _, _, m in mats]),
               norm=_Arena(torch.float32, [m.d_out for _, _, m in mats]),
               sigma=_Arena(torch.float32, [m.d_in // 2 for _, _, m in mats]),
               w_hat=_Arena(torch.bfloat16, [m.d_out * m.d_in for _, _, m in mats]),
               dist=_Arena(torch.float64, [4 for _ in mats]))
    mc = model_codec.ModelCodec(spec, torch.device(DEV, torch.cuda.current_device()), _codebook(K))
    signs = {}
    for i, (layer, mid, m) in enumerate(mats):
        one = seed * 1009 + 16 * layer + mid
        W = synth.make_weight(spec, m, one, device=DEV)
        act = synth.make_act_rms(spec, m.d_in, one, device=DEV)
        if m.d_in not in signs:
            signs[m.d_in] = torch.from_numpy(q.make_signs(q.DEFAULT_SIGN_SEED, m.d_in)).to(DEV)
        scale = torch.from_numpy(q.channel_scales(act.cpu().numpy(), ALPHA)).to(DEV)
        mc.slots.append(model_codec.MatrixSlot(
            f"{layer}.{m.name}", m.d_out, m.d_in, q.make_params(W, m.d_out, m.d_in, case["block"], K), W, act, scale,
            signs[m.d_in], out["sigma"].take(i, (m.d_in // 2,)), out["packed"].take(i, (m.d_out, stride(m))),
            out["norm"].take(i, (m.d_out,)), out["w_hat"].take(i, (m.d_out, m.d_in)), out["dist"].take(i, (4,))))
    mc.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mc.finalize()
    return dict(mc=mc, out={k: v.all for k, v in out.items()})


def prepare(case, seed):
    kind = case["kind"]
    if kind == "model":
        return dict(_model(case, seed), kind=kind)
    if kind == "train":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        return dict(kind=kind, K=case["K"], pairs=torch.randn((case["n"], 2), generator=g, device=DEV, dtype=torch.float64))
    s = dict(_one(case, seed), kind=kind)
    if kind == "quantize":
        return s
    _quantize(s)  # the stream that decode and gemv read
    del s["W"]
    d_out, d_in = case["d_out"], case["d_in"]
    if kind == "decode":
        s["w_hat"] = torch.empty((d_out, d_in), dtype=torch.bfloat16, device=DEV)
    else:
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 1)
        s["x"] = torch.randn((case["n_vec"], d_in), generator=g, device=DEV) * torch.from_numpy(s["act"]).to(DEV)
        s["y"] = torch.empty((d_out, case["n_vec"]), device=DEV)
        s["gemv_ws"] = torch.empty(4 * case["n_vec"] * d_in, dtype=torch.uint8, device=DEV)
    return s


# ------------------------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "quantize":
        _quantize(s)
        return {k: s[k] for k in ("packed", "norm", "sigma", "scale", "signs", "status")}
    if kind == "model":
        s["mc"].step()
        return dict(s["out"], status=s["mc"].status)
    if kind == "decode":
        q.decode(s["packed"], s["norm"], s["scale"], s["signs"], s["sigma"], s["cb"], s["p"], s["w_hat"])
        return s["w_hat"]
    if kind == "gemv":
        q.decode_gemv(s["packed"], s["norm"], s["scale"], s["signs"], s["sigma"], s["cb"], s["p"], s["x"], s["y"], s["gemv_ws"])
        return s["y"]
    out = q.train_codebook_gpu(s["K"], samples=s["pairs"])
    trace = np.zeros(101)  # one error per assignment; inputs differ in how many they take
    trace[:len(out["trace"])] = out["trace"]
    return {"codebook": out["codebook"], "mse": out["mse"], "iters": out["iters"], "trace": trace}


def _shapes(case):
    if case["kind"] == "model":
        layer = synth.decoder_layer(case["hidden"], case["inter"], case["kv"])
        return [(m.d_out, m.d_in) for m in layer] * case["layers"]
    return [(case["d_out"], case["d_in"])]


def work(case):
    """Each input read once, each output written once.  Operations per weight: a rotation's log2(block) additions each
    way, scaling, norm and division (5) for encoding, scaling (3) for decoding, 8 for the distortion sums, 2 per vector for
    a product; a training pass reads every pair once per update and adds it to its cell."""
    kind = case["kind"]
    if kind == "train":
        updates = 100  # the default limit; small codebooks may settle earlier
        return {"bytes": 16 * case["n"] * (updates + 1), "flops": 4 * case["n"] * (updates + 1)}
    w_bytes = 4 if case["dtype"] == "f32" else 2
    stages = int(math.log2(case["block"]))
    total = flops = 0
    for d_out, d_in in _shapes(case):
        n = d_out * d_in
        packed = d_out * ((d_in // 2 * int(math.log2(case["K"])) + 7) // 8 + 4)
        columns = d_in * (4 + 1 + 2)  # channel scale, sign, half a pair scale
        if kind == "quantize":
            total, flops = total + n * w_bytes + packed + columns, flops + n * (5 + stages)
        elif kind == "model":
            total, flops = total + n * (w_bytes + 2) + packed + columns, flops + n * (16 + 2 * stages)
        elif kind == "decode":
            total, flops = total + n * 2 + packed + columns, flops + n * (3 + stages)
        else:
            v = case["n_vec"]
            total, flops = total + packed + columns + 4 * v * (d_in + d_out), flops + 2 * n * v
    return {"bytes": total, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "gemv":
        return {"rel": 1e-5, "max": 1e-4}  # sums in f32
    if kind == "decode":
        return {"rel": 1e-3, "max": 1e-2}  # bf16 weights: some round the other way
    if kind == "model":
        return {"rel": 1e-3, "max": 1e-2, "differ": 1e-6}  # the same, and a pair scale's last bit can move an index
    if kind == "train":
        return {"rel": 1e-6, "max": 1e-5}  # doubles rounded to f32 at the end
    return {"rel": 1e-6, "max": 1e-5, "differ": 1e-6}
