"""What is measured of this framework: the calls a decoding program makes.

Three kinds of call, each through libgs's public entry points (the same-name
binding in ``paper_2609_26638_gb300/gs.py``):

  linear     one projection or LM head of the decoder (``gs_linear``) on the
             decoder's weight shapes: decode windows, serving windows and
             prefill chunks, with the split-K factors the decoder uses
  attention  the paged hybrid-mask attention (``gs_attention``): draft and
             verify windows, batch 1 to 64, and a causal prefill chunk
  decode     whole calls: sequences are (re)started, then forced
             self-speculative rounds run (``gs_round``), the last with both
             heads' logits

Sizes are the repository's own: the GLM-OCR-scale decoder of ``synth.GLM``,
its workloads and the attention sweep.  Inputs come from the seed alone.
"""
import ctypes
import math
import random

import numpy as np
import torch

import synth
from paper_2609_26638_gb300 import gs

DEV = "cuda:0"
SMS = 152              # the split-K rule of the decoder is stated in these
GLM = synth.GLM
D, F, V = GLM.d_model, GLM.d_ffn, GLM.vocab
HQ, HKV = GLM.n_heads, GLM.n_kv_heads
PAGE = 64

# weight shapes of the decoder: output features N, reduction K, epilogue
SHAPES = {
    "qkv": (GLM.qkv_dim, D, "store"),
    "o": (D, HQ * 64, "resid"),
    "gate_up": (F, D, "swiglu"),
    "down": (D, F, "resid"),
    "lm_head": (V, D, "argmax"),
}
EPILOGUE = {"store": gs.EPI_STORE_F16, "resid": gs.EPI_RESID_F32, "swiglu": gs.EPI_SWIGLU,
            "argmax": gs.EPI_ARGMAX}


def decode_split(rows, K):
    """Split-K factor the decoder gives a weight of `rows` x K in decode windows."""
    tiles, nkb = rows // 128, K // 64
    if tiles >= SMS:
        return 1
    want = min(max(-(-SMS // tiles), 4), 8)
    return max(s for s in range(1, want + 1) if nkb % s == 0)


def linear(name, shape, M, decode=True):
    N, K, epi = SHAPES[shape]
    rows = 2 * N if epi == "swiglu" else N
    c = {"kind": "linear", "shape": shape, "M": M, "split": decode_split(rows, K) if decode else 1}
    return {"name": name, **c} if name else c


def attention(name, batch, lo, hi, W, mode, hq=HQ, hkv=HKV):
    c = {"kind": "attention", "batch": batch, "lo": lo, "hi": hi, "W": W, "mode": mode, "hq": hq,
         "hkv": hkv}
    return {"name": name, **c} if name else c


def decode(name, batch, lo, hi, K, rounds, prefill):
    c = {"kind": "decode", "batch": batch, "lo": lo, "hi": hi, "K": K, "rounds": rounds,
         "prefill": prefill}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one document at a time: the attention of a draft window over a 2048-slot prefix
        attention("attn_page_b1", 1, 2048, 2048, 17, "draft"),
        # the serving batch: 32 documents of 1024..6144 slots, ragged, verify windows
        attention("attn_serve_b32", 32, 1024, 6144, 17, "verify"),
        # long dense pages, wide windows: 8 documents of 8192 slots, K = 32
        attention("attn_long_b8", 8, 8192, 8192, 33, "draft"),
        # the widest batch of the attention sweep, short windows: KV streaming
        attention("attn_sweep_b64", 64, 8192, 8192, 9, "draft"),
        # a prefill chunk of 1024 tokens behind 3072 cached ones (causal)
        attention("attn_chunk_1024", 1, 3072, 3072, 1024, "verify"),
        # batch-1 decode window (17 rows): QKV projection, latency of one small GEMM
        linear("lin_qkv_b1", "qkv", 17),
        # serving window (32 x 17 rows): gate/up + SwiGLU and the down projection + residual
        linear("lin_gate_up_serve", "gate_up", 544),
        linear("lin_down_serve", "down", 544),
        # prefill chunk of the default size (4096 tokens): gate/up + SwiGLU
        linear("lin_gate_up_prefill", "gate_up", 4096, decode=False),
        # LM head + argmax of a batch-1 window: the vocabulary streamed once
        linear("lm_head_b1", "lm_head", 17),
        # one request end to end: a 2048-token page prefilled, then eight rounds of K = 16
        decode("page_b1", 1, 2048, 2048, 16, 8, True),
        # serving: four rounds of 32 ragged documents (prefilled beforehand), K = 16
        decode("serve_b32", 32, 1024, 6144, 16, 4, False),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["linear"] * 4 + ["attention"] * 4 + ["decode"])
    if kind == "linear":
        shape = rng.choice(list(SHAPES))
        decoding = shape == "lm_head" or rng.random() < 0.65
        M = _log(rng, 1, 600) if decoding else _log(rng, 100, 4096)
        return linear(None, shape, M, decoding)
    if kind == "attention":
        hq, hkv = rng.choice([(HQ, HKV), (HQ, HKV), (HQ, HKV), (4, 4)])
        if rng.random() < 0.2:    # a prefill chunk
            n = _log(rng, 1, 6000)
            return attention(None, 1, n, n, _log(rng, 100, 1024), "verify", hq, hkv)
        hi = _log(rng, 256, 8192)
        lo = rng.choice([hi, rng.randint(1, hi)])
        return attention(None, _log(rng, 1, 64), lo, hi, 1 + _log(rng, 1, 64),
                         rng.choice(["draft", "verify"]), hq, hkv)
    batch = _log(rng, 1, 8)
    hi = _log(rng, 128, 4096)
    return decode(None, batch, max(1, hi // 3) if batch > 1 else hi, hi, rng.randint(1, 32),
                  rng.randint(1, 4), rng.random() < 0.5)


def _lengths(c, seed):
    rng = random.Random(seed * 7919 + 11)
    return [rng.randint(c["lo"], c["hi"]) for _ in range(c["batch"])]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


# ------------------------------------------------------------------ linear
class _Linear:
    """Inputs of one gs_linear call and the scratch its caller keeps."""

    def __init__(self, c, seed):
        self.M, self.split = c["M"], c["split"]
        self.N, self.K, epi = SHAPES[c["shape"]]
        self.epi_name, self.epi = epi, EPILOGUE[epi]
        g = _gen(seed)
        rows = 2 * self.N if epi == "swiglu" else self.N
        self.x = torch.randn(self.M, self.K, device=DEV, generator=g).half()
        self.w = (synth.WEIGHT_STD * torch.randn(rows, self.K, device=DEV, generator=g)).half()
        if epi == "resid":     # the residual stream the call adds to
            self.y = torch.randn(self.M, self.N, device=DEV, generator=g)
        elif epi == "argmax":
            self.y = torch.zeros(self.M, dtype=torch.int64, device=DEV)
        else:
            self.y = torch.zeros(self.M, self.N, dtype=torch.float16, device=DEV)
        self.sb = gs.gs_linear_scratch_bytes(self.M, self.N, self.split)
        self.scratch = torch.zeros(self.sb, dtype=torch.uint8, device=DEV)

    def run(self):
        if self.epi_name == "argmax":
            self.y.zero_()     # the keys are combined with a maximum: the caller clears them
        gs.gs_linear(self.x.data_ptr(), self.w.data_ptr(), self.y.data_ptr(), self.M, self.N,
                     self.K, self.epi, self.split, self.scratch.data_ptr(), self.sb,
                     torch.cuda.current_stream().cuda_stream)
        return self.y

    def exact(self):
        if self.epi_name == "argmax":
            return None
        acc = self.x.double() @ self.w.double().T
        if self.epi_name == "resid":
            return self.y.double() + acc
        if self.epi_name == "swiglu":
            gate, up = acc[:, :self.N], acc[:, self.N:]
            return gate / (1 + torch.exp(-gate)) * up
        return acc


# ------------------------------------------------------------------ attention
class _Attention:
    """A paged pool with every sequence's keys and values in shuffled pages."""

    def __init__(self, c, seed):
        self.B, self.W, self.hq, self.hkv = c["batch"], c["W"], c["hq"], c["hkv"]
        self.mode = gs.ATTN_VERIFY if c["mode"] == "verify" else gs.ATTN_DRAFT
        self.ns = _lengths(c, seed)
        pages = [(n + self.W + 1 + PAGE - 1) // PAGE for n in self.ns]
        self.n_pages, self.stride = sum(pages), max(pages)
        perm = np.random.default_rng(seed).permutation(self.n_pages).astype(np.int32)
        pt = np.full((self.B, self.stride), -1, np.int32)
        at = 0
        for b, p in enumerate(pages):
            pt[b, :p] = perm[at:at + p]
            at += p
        g = _gen(seed)
        # fp16 N(0, 1), as the sweep's keys, values and queries
        self.kv = torch.empty(self.n_pages, 2, self.hkv, 64, 64, dtype=torch.float16, device=DEV)
        self.kv.normal_(generator=g)
        self.q = torch.randn(self.B, self.W, self.hq, 64, device=DEV, generator=g).half()
        self.out = torch.zeros_like(self.q)
        self.pt = torch.from_numpy(pt).to(DEV)
        self.n = torch.tensor(self.ns, dtype=torch.int32, device=DEV)
        # pages per work item as the engine sets them: at most 16 items per
        # sequence when a batch of them fits about one wave of CTAs, else 8
        blocks = self.B * -(-self.W // min(self.W, 128 // (self.hq // self.hkv)))
        items = 16 if blocks * self.hkv * 16 <= 2 * SMS else 8
        self.sp = max(2, -(-self.stride // items))
        self.sb = gs.gs_attention_scratch_bytes(self.B, self.W, self.hq, self.hkv, self.stride,
                                                self.sp)
        self.scratch = torch.zeros(self.sb, dtype=torch.uint8, device=DEV)

    def run(self):
        gs.gs_attention(self.mode, self.q.data_ptr(), self.kv.data_ptr(), self.n_pages,
                        self.pt.data_ptr(), self.stride, self.n.data_ptr(), self.B, self.W,
                        self.hq, self.hkv, self.out.data_ptr(), self.scratch.data_ptr(), self.sb,
                        self.sp, torch.cuda.current_stream().cuda_stream)
        return self.out

    def exact(self):
        G = self.hq // self.hkv
        out = torch.empty(self.B, self.W, self.hq, 64, dtype=torch.float64, device=DEV)
        i = torch.arange(self.W, device=DEV)
        for b, n in enumerate(self.ns):
            if self.mode == gs.ATTN_DRAFT:
                lim = torch.where(i == 0, n, n + self.W - 1)
            else:
                lim = n + 1 + i
            keys = int(lim.max()) + 1
            used = self.kv[self.pt[b, :-(-keys // PAGE)].long()].double()    # [pages, 2, hkv, 64, 64]
            k = used[:, 0].permute(1, 0, 2, 3).reshape(self.hkv, -1, 64)[:, :keys]
            v = used[:, 1].permute(1, 0, 3, 2).reshape(self.hkv, -1, 64)[:, :keys]
            q = self.q[b].double().reshape(self.W, self.hkv, G, 64).permute(1, 2, 0, 3)
            s = q.reshape(self.hkv, G * self.W, 64) @ k.transpose(1, 2) / 8.0
            hidden = torch.arange(keys, device=DEV)[None, :] > lim[:, None]
            s = s.reshape(self.hkv, G, self.W, keys).masked_fill(hidden, -math.inf)
            o = torch.softmax(s, dim=-1).reshape(self.hkv, G * self.W, keys) @ v
            out[b] = o.reshape(self.hkv, G, self.W, 64).permute(2, 0, 1, 3).reshape(self.W, self.hq, 64)
        return out


# ------------------------------------------------------------------ decode
# A trained decoder's next token is clear of the second best; random heads are
# not, and their argmax would follow the last bit.  So the embedding is N(0, 1)
# and the LM head holds, for every token, the embedding of its predecessor in a
# fixed cycle over the vocabulary: the greedy continuation is that cycle.
_streams = []


def _stream():
    """The one stream a decoding program gives its handles (graphs need a non-default one)."""
    if not _streams:
        _streams.append(torch.cuda.Stream(DEV))
    return _streams[0]


class _Decode:
    def __init__(self, c, seed, engine=True):
        self.c, self.B, self.K = c, c["batch"], c["K"]
        self.lengths = _lengths(c, seed)
        g = _gen(seed)

        def normal(rows, cols, std):
            w = torch.empty(rows, cols, dtype=torch.bfloat16, device=DEV).normal_(generator=g)
            return w.mul_(std)

        self.shift = 1 + seed % (V - 3)
        self.embed = normal(V, D, 1.0)
        self.lm_head = torch.roll(self.embed, self.shift, 0).mul_(synth.WEIGHT_STD)
        self.ones = torch.ones(D, dtype=torch.bfloat16, device=DEV)
        self.layers = [{"w_qkv": normal(GLM.qkv_dim, D, 0.02), "w_o": normal(D, HQ * 64, 0.02),
                        "w_gate_up": normal(2 * F, D, 0.02), "w_down": normal(D, F, 0.02)}
                       for _ in range(GLM.n_layers)]
        rng = np.random.default_rng(seed)
        self.vis, self.text, self.x0 = [], [], []
        for P in self.lengths:     # 75 % visual rows, then prompt tokens
            n_text = max(1, P // 4)
            self.vis.append(normal(P - n_text, D, 1.0))
            t = rng.integers(0, V - 1, n_text).astype(np.int32)
            self.text.append(torch.from_numpy(t).to(DEV))
            self.x0.append(int((t[-1] + self.shift) % V))
        R, K = c["rounds"], self.K
        # accepted lengths: censored geometric, mean about 0.6 K (9.7 of 16)
        alpha = synth.solve_alpha(0.606 * K, K)
        u = np.maximum(rng.random((self.B, R)), 1e-12)
        self.L = np.minimum(np.floor(np.log(u) / math.log(alpha)), K).astype(np.int32)
        self.max_new = R * (K + 2) + 2
        ctx = max(self.lengths) + self.max_new + K + 2
        # greedy continuation by absolute slot; teacher[P] is the boundary token
        slot = np.arange(ctx)[None, :] - np.array(self.lengths)[:, None]
        self.teacher = np.where(slot >= 0, (np.array(self.x0)[:, None] + slot * self.shift) % V, 0)
        self.h = None
        if engine:
            self._create(ctx)

    def _create(self, ctx):
        c = gs.gs_config()
        for f in ("n_layers", "d_model", "n_heads", "n_kv_heads", "head_dim", "d_ffn", "vocab",
                  "rope_theta", "rms_eps", "mask_token_id"):
            setattr(c, f, getattr(GLM, f))
        c.eos_token_id = -1
        c.max_batch, c.max_ctx, c.max_K, c.max_prefill = self.B, ctx, self.K, 4096
        c.kv_pages = sum(-(-(P + self.max_new + self.K + 2) // PAGE) for P in self.lengths)
        c.split_pages = 0
        w = gs.gs_weights()
        w.embed, w.lm_head = self.embed.data_ptr(), self.lm_head.data_ptr()
        w.final_norm = self.ones.data_ptr()
        L = GLM.n_layers
        arr = ctypes.c_void_p * L
        norm = arr(*[self.ones.data_ptr()] * L)
        self._keep = [norm]
        w.attn_norm = w.ffn_norm = ctypes.cast(norm, ctypes.POINTER(ctypes.c_void_p))
        for f in ("w_qkv", "w_o", "w_gate_up", "w_down"):
            a = arr(*[lw[f].data_ptr() for lw in self.layers])
            self._keep.append(a)
            setattr(w, f, ctypes.cast(a, ctypes.POINTER(ctypes.c_void_p)))
        self.ws = torch.empty(gs.gs_workspace_bytes(c), dtype=torch.uint8, device=DEV)
        self.stream = _stream()
        torch.cuda.synchronize()
        self.h = gs.gs_create(c, w, self.ws.data_ptr(), self.ws.numel(), self.stream.cuda_stream)
        K, B = self.K, self.B
        i32 = dict(dtype=torch.int32, device=DEV)
        self.slots = torch.arange(B, **i32)
        self.tok, self.cnt, self.done = (torch.zeros(B, K + 2, **i32), torch.zeros(B, **i32),
                                         torch.zeros(B, **i32))
        self.x0_out = torch.zeros(B, **i32)
        self.teacher_d = torch.from_numpy(self.teacher.astype(np.int32)).to(DEV)
        self.L_d = torch.from_numpy(self.L).to(DEV)
        self.force = gs.gs_force()
        self.force.teacher, self.force.teacher_stride = self.teacher_d.data_ptr(), self.teacher.shape[1]
        self.force.L_sched, self.force.L_stride = self.L_d.data_ptr(), self.L.shape[1]
        self.logits = [torch.zeros(B, K + 1, V, device=DEV) for _ in range(2)]
        self.dbg = gs.gs_debug()
        self.dbg.draft_logits, self.dbg.verify_logits = (t.data_ptr() for t in self.logits)
        torch.cuda.synchronize()
        if not self.c["prefill"]:
            self._prefill()
            torch.cuda.synchronize()

    def _prefill(self):
        for s in range(self.B):
            vis, text = self.vis[s], self.text[s]
            gs.gs_prefill(self.h, s, vis.data_ptr() if vis.shape[0] else 0, vis.shape[0],
                          text.data_ptr(), text.shape[0], self.max_new,
                          self.x0_out[s:].data_ptr())

    def run(self):
        if self.c["prefill"]:
            self._prefill()
        else:      # every sequence back to the end of its prefix
            for s, P in enumerate(self.lengths):
                gs.gs_seq_restore(self.h, s, P, self.x0[s], 1, self.max_new, 0, 0)
        args = (self.h, self.slots.data_ptr(), self.B, self.K, gs.GS_ACCEPT_GREEDY, self.force,
                self.tok.data_ptr(), self.cnt.data_ptr(), self.done.data_ptr())
        for _ in range(self.c["rounds"] - 1):
            gs.gs_round(*args)
        gs.gs_round(*args, self.dbg)
        return {"x0": self.x0_out, "tok": self.tok, "cnt": self.cnt, "done": self.done,
                "draft_logits": self.logits[0], "verify_logits": self.logits[1]}

    def __del__(self):
        if getattr(self, "h", None) is not None:
            self.stream.synchronize()
            gs.gs_destroy(self.h)
            self.h = None

    def exact(self):
        """The last round's logits: per sequence one forward in 64 bits over
        [prefix, committed tokens, x0, a0, d_1..d_K] (causal) and the K mask
        rows of the draft window (they see slots 0..n and one another)."""
        draft, verify = [], []
        for b, P in enumerate(self.lengths):
            n = P + int((self.L[b, :-1] + 2).sum())         # cached slots at the last round
            tch, K, L = self.teacher[b], self.K, int(self.L[b, -1])
            win = [int(tch[n + 1 + i]) for i in range(K + 1)]     # a0, d_1..d_K
            if L < K:
                win[L + 1] = (win[L + 1] + 1) % V
                # drafts past the forced ones are the draft rows' own argmax
                mask_next = (GLM.mask_token_id + self.shift) % V
                for i in range(L + 2, K + 1):
                    win[i] = mask_next
            toks = [int(t) for t in tch[P:n + 1]] + win + [GLM.mask_token_id] * K
            ids = torch.cat([self.text[b].long(), torch.tensor(toks, device=DEV)])
            h = torch.cat([self.vis[b].double(), self.embed[ids].double()])
            pos = torch.cat([torch.arange(n + K + 2, device=DEV),
                             torch.arange(n + 1, n + K + 1, device=DEV)])
            T, main = h.shape[0], n + K + 2
            i = torch.arange(T, device=DEV)
            allowed = (i[None, :] <= i[:, None]) & (i[None, :] < main)
            allowed[main:] = (i[None, :] <= n) | (i[None, :] >= main)
            out = self._forward64(h, pos, allowed)
            logits = out[[n, *range(main, T), *range(n + 1, main)]] @ self.lm_head.double().T
            draft.append(logits[:K + 1])
            verify.append(logits[K + 1:])
        return {"x0": None, "tok": None, "cnt": None, "done": None,
                "draft_logits": torch.stack(draft), "verify_logits": torch.stack(verify)}

    def _forward64(self, h, pos, allowed):
        T, G = h.shape[0], HQ // HKV
        ang = pos.double()[:, None] * GLM.rope_theta ** (
            -torch.arange(32, device=DEV, dtype=torch.float64) / 32)
        cos, sin = torch.cos(ang)[:, None], torch.sin(ang)[:, None]

        def rope(x):
            a, b = x[..., :32], x[..., 32:]
            return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

        def norm(x):
            return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + GLM.rms_eps)

        for lw in self.layers:
            qkv = norm(h) @ lw["w_qkv"].double().T
            q = rope(qkv[:, :HQ * 64].reshape(T, HQ, 64))
            k = rope(qkv[:, HQ * 64:(HQ + HKV) * 64].reshape(T, HKV, 64))
            v = qkv[:, (HQ + HKV) * 64:].reshape(T, HKV, 64)
            a = torch.empty(T, HQ, 64, dtype=torch.float64, device=DEV)
            for head in range(HQ):
                s = (q[:, head] @ k[:, head // G].T / 8.0).masked_fill(~allowed, -math.inf)
                a[:, head] = torch.softmax(s, -1) @ v[:, head // G]
            h = h + a.reshape(T, HQ * 64) @ lw["w_o"].double().T
            gu = norm(h) @ lw["w_gate_up"].double().T
            gate, up = gu[:, :F], gu[:, F:]
            h = h + (gate / (1 + torch.exp(-gate)) * up) @ lw["w_down"].double().T
        return norm(h)


# ------------------------------------------------------------------ interface
_KINDS = {"linear": _Linear, "attention": _Attention, "decode": _Decode}


def prepare(case, seed):
    return _KINDS[case["kind"]](case, seed)


def run(state):
    return state.run()


def exact(case, seed):
    if case["kind"] == "decode":
        # 64-bit forwards of one or two pages are quick; a batch of them is not
        if case["batch"] * case["hi"] > 6000:
            return None
        return _Decode(case, seed, engine=False).exact()
    return _KINDS[case["kind"]](case, seed).exact()


def work(case):
    if case["kind"] == "linear":
        N, K, epi = SHAPES[case["shape"]]
        M, rows = case["M"], 2 * N if epi == "swiglu" else N
        out = {"store": 2 * M * N, "swiglu": 2 * M * N, "resid": 8 * M * N, "argmax": 8 * M}[epi]
        return {"bytes": 2 * rows * K + 2 * M * K + out, "flops": 2 * M * rows * K}
    mean = (case["lo"] + case["hi"]) / 2
    if case["kind"] == "attention":
        B, W, hq, hkv = case["batch"], case["W"], case["hq"], case["hkv"]
        keys = mean + W + (1 if case["mode"] == "verify" else 0)
        seen = mean + W / 2 if case["mode"] == "verify" else mean + W
        return {"bytes": B * keys * hkv * 256 + 4 * B * W * hq * 64,
                "flops": 4 * B * W * seen * hq * 64}
    B, K, R = case["batch"], case["K"], case["rounds"]
    layer = GLM.qkv_dim * D + D * HQ * 64 + 3 * F * D
    body, head = GLM.n_layers * layer, V * D
    kv_slot = GLM.n_layers * 2 * HKV * 64 * 2
    rows = B * (K + 1)
    attn = 4 * GLM.n_layers * HQ * 64
    nbytes = 2 * R * (2 * (body + head) + B * mean * kv_slot) + 2 * rows * V * 4
    flops = 2 * R * (2 * rows * (body + head) + attn * rows * mean)
    if case["prefill"]:
        nbytes += B * (2 * (body + head) + mean * (2 * D + kv_slot))
        flops += B * (2 * mean * body + 2 * head + attn * mean * mean / 2)
    return {"bytes": nbytes, "flops": flops}
