"""The work a speculative ASR decoder has this library do, as cases to time.

Every case is one pass through the public entry points (``Session``,
``DraftModel`` and the C ABI's binding) on inputs that already sit on the GPU,
as in a decoding loop that never leaves it:

  verify  one verification round of a running batch: the committed state is
          put back (``asr_spec_rollback``, as after a round that is not kept)
          and the draft block scored, accepted and anchored
  score   the same round with the logits of every scored row read back
          (``asr_spec_debug_logits``): rescoring a block of known tokens
  tree    one verification round over a candidate tree per utterance
  start   new audio arrives: encoder K/V cache, prompt prefill, first round
  loop    two rounds of the cached loop: the one-block draft proposes, the
          target verifies, the draft catches up and proposes again

Models are the decoder shapes of the synthetic workloads (tiny in fp32, small
and large in bf16); layers are cut in most cases so that a state is made
quickly, the widths and the vocabulary never.  Ranges: 1 to 64 utterances, up to
16 drafts, 100 to 3000 encoder frames, prompts of 1 to 224 tokens (a fixed
header up to a previous segment's text).

Weights follow a trained decoder in the two respects that decide discrete
results: the token embedding outweighs the residual branches (output
projections scaled by 1 / sqrt(2 layers)), so that argmax decisions have
margins, and the anchor layer's cross-attention has a clear audio peak (its
query bias points at one frame per utterance).  The greedy continuation of
such a model repeats the pending token, so a draft block's accepted length is
known when it is made.
"""
import math
import types

import numpy as np
import torch

from paper_2608_12703_gb300 import asrspec as A
from paper_2608_12703_gb300.session import DraftModel, Session

MAX_POS = 448
MODELS = {   # d_model, heads, feed-forward, vocabulary, storage
    "tiny": (384, 6, 1536, 51865, "fp32"),
    "small": (768, 12, 3072, 51865, "bf16"),
    "large": (1280, 20, 5120, 51866, "bf16"),
}
FULL_LAYERS = {"tiny": 4, "small": 12, "large": 32}


def case(kind, model, layers, batch, k, frames, frames_min=0, prompt=4, threshold=0.0):
    return {"kind": kind, "model": model, "layers": layers, "batch": batch, "k": k, "frames": frames,
            "frames_min": frames_min or frames, "prompt": prompt, "threshold": threshold}


def listed():
    return [
        # the smallest call: the fp32 decoder, one 30 s utterance, mid-transcript
        dict(case("verify", "tiny", 4, 1, 4, 1500, prompt=32), name="verify tiny fp32 b1 k4"),
        # the latency of one stream on the full large decoder (every layer)
        dict(case("verify", "large", 32, 1, 8, 1500, prompt=112), name="verify large full b1 k8"),
        # a few concurrent streams of mixed length: too many rows for one, too few for a batch
        dict(case("verify", "large", 8, 5, 6, 1417, 389, prompt=60), name="verify large b5 k6"),
        # a server's batch: 64 utterances of 5 to 30 s, a tenth of them done
        dict(case("verify", "large", 8, 64, 6, 1500, 250, prompt=31), name="verify large b64 k6"),
        # the small decoder with the longest blocks
        dict(case("verify", "small", 12, 32, 16, 1500, prompt=64), name="verify small full b32 k16"),
        # rescoring known blocks, logits wanted
        dict(case("score", "small", 12, 3, 9, 1100, 713, prompt=20), name="score small full b3 k9"),
        # an 11-node candidate tree on one stream
        dict(case("tree", "large", 8, 1, 11, 1500, prompt=112), name="tree large b1 n11"),
        # one new utterance
        dict(case("start", "large", 8, 1, 8, 1500), name="start large b1"),
        # a batch of new utterances (the most work)
        dict(case("start", "large", 8, 64, 6, 1500, 250), name="start large b64"),
        # new audio that carries its previous segment's text as prompt
        dict(case("start", "small", 12, 4, 7, 1500, 901, prompt=203), name="start small full b4 prompt 203"),
        # the cached loop on one stream
        dict(case("loop", "large", 4, 1, 8, 1500, prompt=40), name="loop large b1 k8"),
        # the cached loop on a batch
        dict(case("loop", "small", 12, 24, 4, 1500, 640, prompt=23), name="loop small full b24 k4"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["verify", "verify", "verify", "score", "tree", "start", "start", "loop", "loop"])
    model = rng.choice(["tiny", "small", "large", "large"] if kind in ("verify", "score", "start") else
                       ["small", "large"])
    layers = {"tiny": 4, "small": rng.randint(4, 12), "large": rng.randint(4, 8)}[model]
    k = rng.randint(1, 16)
    batch = _log(rng, 1, {"tiny": 16, "small": 64, "large": 64}[model])
    batch = min(batch, {"score": 8, "start": 34}.get(kind, 64))
    batch = max(1, min(batch, 560 // (k + 1)))
    prompt = _log(rng, 1, 224 if batch <= 16 else 8 if kind == "start" else 96)
    frames = rng.randint(1501, 3000) if batch <= 4 and rng.random() < 0.15 else rng.randint(100, 1500)
    return case(kind, model, layers, batch, k, frames, rng.randint(min(100, frames), frames),
                prompt, rng.choice([0.0, 0.0, 0.3]) if kind == "loop" else 0.0)


# ---- shapes of a case (the same for every seed) --------------------------------

def _frames(c):
    """Encoder frames per utterance, spread over [frames_min, frames]; the first has the most."""
    lo, hi = c["frames_min"], c["frames"]
    return [hi if b == 0 else lo + (b * 7919 + 13) % 1000 * (hi - lo) // 999 for b in range(c["batch"])]


def _lens(c):
    """Drafts per utterance: whole blocks, shorter ones near an end, and in a batch some that have finished (-1)."""
    B, k = c["batch"], c["k"]
    if B < 4:
        return [k] * B
    return [-1 if b % 10 == 7 else (k + 1) // 2 if b % 3 == 1 else k for b in range(B)]


# ---- weights ---------------------------------------------------------------------

def _layer_shapes(d, f):
    return [("ln1_g", (d,)), ("ln1_b", (d,)), ("wq", (d, d)), ("bq", (d,)), ("wk", (d, d)), ("wv", (d, d)),
            ("bv", (d,)), ("wo", (d, d)), ("bo", (d,)), ("ln2_g", (d,)), ("ln2_b", (d,)), ("wcq", (d, d)),
            ("bcq", (d,)), ("wck", (d, d)), ("wcv", (d, d)), ("bcv", (d,)), ("wco", (d, d)), ("bco", (d,)),
            ("ln3_g", (d,)), ("ln3_b", (d,)), ("w1", (f, d)), ("b1", (f,)), ("w2", (d, f)), ("b2", (d,))]


def _views(flat, shapes):
    out, at = {}, 0
    for name, shape in shapes:
        n = math.prod(shape)
        out[name] = flat[at:at + n].view(shape)
        at += n
    assert at == flat.numel()
    return out


def _normal(shapes, seed, dtype):
    """0.02 N(0, 1) in every entry, gains 1 + that, rounded to the storage type."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(dev).manual_seed(seed)
    flat = torch.empty(sum(math.prod(s) for _, s in shapes), device=dev).normal_(0.0, 0.02, generator=g)
    w = _views(flat, shapes)
    for name in w:
        if name.endswith("_g"):
            w[name] += 1.0
    return flat, w, (lambda t: t.copy_(t.bfloat16())) if dtype == "bf16" else (lambda t: t)


def _target_shapes(c):
    d, _, f, v, _ = MODELS[c["model"]]
    s = [("tok_emb", (v, d)), ("pos_emb", (MAX_POS, d))]
    for l in range(c["layers"]):
        s += [("%d.%s" % (l, n), shape) for n, shape in _layer_shapes(d, f)]
    return s + [("lnf_g", (d,)), ("lnf_b", (d,))]


def _anchor_layer(c):
    return 3 * c["layers"] // 4


def _peak_state(c):
    """The encoder state that the anchor layer's heads look for, N(0, 1) entries."""
    d = MODELS[c["model"]][0]
    u = torch.from_numpy(np.random.default_rng(11).standard_normal(d).astype(np.float32))
    return u.bfloat16().float() if MODELS[c["model"]][4] == "bf16" else u


def _target_weights(c):
    """The decoder's parameters: one flat fp32 tensor in the library's order, and its parts."""
    flat, w, store = _normal(_target_shapes(c), 0, MODELS[c["model"]][4])
    w["tok_emb"] *= 25.0
    for l in range(c["layers"]):
        for n in ("wo", "wco", "w2"):
            w["%d.%s" % (l, n)] /= math.sqrt(2.0 * c["layers"])
    a = _anchor_layer(c)
    store(flat)
    w["%d.bcq" % a].copy_(w["%d.wck" % a] @ _peak_state(c).to(flat.device))
    return flat, w


def _draft_weights(c):
    """The one-block draft's parameters; its input combination is small beside the token embedding."""
    d = MODELS[c["model"]][0]
    flat, w, store = _normal([("w_in", (d, 4 * d)), ("b_in", (d,))] + _layer_shapes(d, 2 * d) +
                             [("lnf_g", (d,)), ("lnf_b", (d,))], 5, "bf16")
    w["w_in"] /= 4.0
    for n in ("wo", "wco", "w2"):
        w[n] /= 2.0
    store(flat)
    return flat


_blob = {}   # the one model whose host parameters are at hand, as a server has its checkpoint


def _host_blob(c):
    key = (c["model"], c["layers"])
    if key not in _blob:
        _blob.clear()
        _blob[key] = _target_weights(c)[0].cpu().numpy()
    return _blob[key]


# ---- inputs ----------------------------------------------------------------------

def _inputs(c, seed):
    """Encoder states [B][T][d] with the peak frame planted, prompts, and the draft block of a round."""
    d, _, _, v, dtype = MODELS[c["model"]]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    B, k, P0 = c["batch"], c["k"], c["prompt"]
    rng = np.random.default_rng([seed, 7])
    g = torch.Generator(dev).manual_seed(seed)
    enc = torch.empty((B, c["frames"], d), device=dev).normal_(generator=g)
    peak = _peak_state(c).to(dev)
    for b, t in enumerate(_frames(c)):
        enc[b, int(rng.integers(0, t))] = peak
    enc = enc.bfloat16() if dtype == "bf16" else enc
    prompt = rng.integers(0, v, (B, P0)).astype(np.int32)
    # greedy repeats the pending token: a prefix of each block is accepted, then a token is wrong
    lens = np.array(_lens(c), np.int32)
    block = rng.integers(0, v - 1, (B, k)).astype(np.int32)
    block += block >= prompt[:, -1:]          # never the pending token
    for b in range(B):
        if lens[b] > 0:
            block[b, :int(rng.integers(0, lens[b] + 1))] = prompt[b, -1]
    # a tree: every node's parent at random; the pending token on about half the nodes
    parent = np.stack([rng.integers(0, np.arange(1, k + 1)) for _ in range(B)]).astype(np.int32)
    nodes = np.where(rng.random((B, k)) < 0.5, prompt[:, -1:], block).astype(np.int32)
    return enc, prompt, lens, block, parent, nodes


def _total_len(c):
    """Transcript lengths for the drafted loop: finished for the utterances that sit out, else long enough."""
    return [c["prompt"] if n < 0 else MAX_POS for n in _lens(c)]


def prepare(c, seed):
    d, heads, f, v, dtype = MODELS[c["model"]]
    B, k = c["batch"], c["k"]
    dims = types.SimpleNamespace(n_layers=c["layers"], d_model=d, n_heads=heads, d_ffn=f, vocab=v, max_pos=MAX_POS,
                                 max_enc=c["frames"], dtype=dtype, anchor_layer=-1)
    enc, prompt, lens, block, parent, nodes = _inputs(c, seed)
    s = types.SimpleNamespace(kind=c["kind"], k=k, prompt_len=c["prompt"], frames=c["frames"], enc=enc, draft=None)
    s.sess = Session(dims, _host_blob(c), max_batch=B, max_draft=k)
    if c["kind"] == "loop":
        s.draft = DraftModel(s.sess, _draft_weights(c).cpu().numpy(), _total_len(c), k, "anchor", c["threshold"])
    dev = enc.device

    def on_gpu(a):
        return torch.from_numpy(np.ascontiguousarray(np.asarray(a, np.int32))).to(dev)

    s.enc_lens, s.prompt = on_gpu(_frames(c)), on_gpu(prompt)
    s.block, s.lens, s.parent, s.nodes = on_gpu(block), on_gpu(lens), on_gpu(parent), on_gpu(nodes)
    s.kv, s.pending = on_gpu([c["prompt"] - 1] * B), on_gpu(prompt[:, -1])
    s.path = torch.zeros((B, k), dtype=torch.int32, device=dev)
    s.profile = torch.zeros((B, c["frames"]), device=dev)
    active = s.lens >= 0
    s.real = (torch.arange(c["frames"], device=dev)[None, :] < s.enc_lens[:, None]) & active[:, None]
    s.seen = torch.zeros_like(s.profile)
    s.zero = torch.zeros((), device=dev)
    s.rows = int(sum(n + 1 for n in _lens(c)))
    s.logits = torch.zeros((s.rows, v), device=dev) if c["kind"] == "score" else None
    torch.cuda.synchronize()
    if c["kind"] != "start":
        _start(s)
        s.sess.stream.synchronize()
    return s


# ---- a pass ------------------------------------------------------------------------

def _start(s):
    A.asr_spec_encode_cache(s.sess.h, s.enc.shape[0], s.enc, s.frames, s.enc_lens)
    s.sess.B = s.enc.shape[0]
    A.asr_spec_prefill(s.sess.h, s.prompt, s.prompt_len)


def _attention_profile(s):
    """The audio attention behind the anchors, real frames of the active utterances."""
    A.asr_spec_debug_anchor_profile(s.sess.h, s.profile)
    return torch.where(s.real, s.profile, s.zero, out=s.seen)


def run(s):
    # inputs come from the caller's stream and results go back to it, so passes follow one another
    caller = torch.cuda.current_stream()
    s.sess.stream.wait_stream(caller)
    with torch.cuda.stream(s.sess.stream):
        out = _pass(s)
    caller.wait_stream(s.sess.stream)
    return out


def _pass(s):
    h = s.sess.h
    if s.kind == "start":
        _start(s)
    else:
        A.asr_spec_rollback(h, s.kv, s.pending)
    if s.kind == "tree":
        o = s.sess.out[:, :s.sess.B]
        A.asr_spec_verify_tree(h, s.nodes, s.parent, s.lens, s.k, o[0], o[1], o[2], o[3], s.path)
        return {"step": o[:4], "path": s.path, "profile": _attention_profile(s)}
    if s.kind == "loop":
        rounds = []
        for _ in range(2):
            d, l = s.draft.propose()
            rounds.append(torch.cat([l[None], s.sess.verify_device(d, l, s.k)[:4]]))   # the tokens a caller keeps
        return {"rounds": rounds, "profile": _attention_profile(s)}
    o = s.sess.verify_device(s.block, s.lens, s.k)[:4]
    if s.kind == "score":
        n = A.asr_spec_debug_logits(h, s.logits, s.rows)
        return {"step": o, "profile": _attention_profile(s), "logits": s.logits[:n]}
    return {"step": o, "profile": _attention_profile(s)}


# ---- what a pass cannot do without ---------------------------------------------------

def work(c):
    d, _, f, v, dtype = MODELS[c["model"]]
    L, B, k, P = c["layers"], c["batch"], c["k"], c["prompt"] - 1
    es = 2 if dtype == "bf16" else 4
    frames, lens = _frames(c), _lens(c)
    on = [b for b in range(B) if lens[b] >= 0]
    per_row = L * (6 * d * d + 2 * f * d)   # projection multiply-adds of one row in the layers

    def layers(rows, keys, utterances):
        """Layer weights once, the cached keys and values of the utterances once."""
        audio = sum(frames[b] for b in utterances)
        by = (per_row + L * 2 * d * (keys * len(utterances) + audio)) * es
        fl = 2 * rows * per_row + 4 * d * L * rows * (keys + audio / max(1, len(utterances)))
        return by, fl

    def verify(rows, keys):
        by, fl = layers(rows, keys, on)
        return by + (v * d + d * sum(frames[b] for b in on)) * es, fl + 2 * rows * v * d

    if c["kind"] == "loop":
        by = fl = 0.0
        n = len(on)
        for i in range(2):   # the block's weights and the tied head once per proposal, then the round's verification
            rows = n * (k + (k if i else 0))
            by += k * (14 * d * d + v * d) * es
            fl += 2 * (rows * 14 * d * d + n * k * v * d)
            b2, f2 = verify(n * (k + 1), P + i * (k + 1))
            by, fl = by + b2, fl + f2
        return {"bytes": by, "flops": fl}
    by, fl = verify(sum(lens[b] + 1 for b in on), P)
    if c["kind"] == "score":
        by += sum(lens[b] + 1 for b in on) * v * 4
    if c["kind"] == "start":
        audio = sum(frames)
        by += audio * d * es + L * 2 * d * d * es + L * 2 * d * audio * es   # states and weights in, K/V out
        fl += 2 * audio * 2 * d * d * L
        if P > 0:
            b2, f2 = layers(B * P, 0, range(B))
            by, fl = by + b2, fl + f2
    return {"bytes": by, "flops": fl}


def tolerance(c):
    """About four times the error against 64 bits, which is 8e-8 (profile) to 4e-7 (logits) in fp32, and 4e-4 to
    2.5e-3 with bf16 operands through 4 to 32 layers (the logits have the most).  Tokens, lengths and frames are decided with
    margins and stay the same."""
    if MODELS[c["model"]][4] == "fp32":
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.0}
    return {"rel": 1e-2, "max": 0.05, "differ": 0.0}


# ---- the same in 64 bits ----------------------------------------------------------------

def _ln(x, g, b):
    return torch.nn.functional.layer_norm(x, (x.shape[-1],), g.double(), b.double(), 1e-5)


def exact(c, seed):
    d, heads, f, v, _ = MODELS[c["model"]]
    L, B, k, P0 = c["layers"], c["batch"], c["k"], c["prompt"]
    frames = _frames(c)
    if 4e0 * sum(frames) * d * d * L > 1.2e13:
        return None
    enc, prompt, lens, block, parent, nodes = _inputs(c, seed)
    _, w = _target_weights(c)
    dev = enc.device
    dt = torch.float64
    loop = c["kind"] == "loop"
    seqs, poss, masks, firsts = [], [], [], []
    for b in range(B):   # every row an utterance has: its committed tokens, then the block (or the tree's nodes)
        n = max(int(lens[b]), 0)
        tail = nodes[b, :n] if c["kind"] == "tree" else block[b, :n]
        if loop:
            n = 0 if lens[b] < 0 else 2 * k + 1
            tail = np.full(n, prompt[b, -1])
        m = P0 + n
        vis = np.tril(np.ones((m, m), bool))
        pos = np.arange(m)
        if c["kind"] == "tree":
            for i in range(1, n + 1):
                r = P0 - 1 + i
                vis[r, P0 - 1:] = False
                p = P0 - 1 + int(parent[b, i - 1])
                vis[r, P0 - 1:] |= vis[p, P0 - 1:]
                if p == P0 - 1:
                    vis[r, p] = True
                vis[r, r] = True
                pos[r] = pos[p] + 1
        seqs.append(np.concatenate([prompt[b], tail]).astype(np.int64))
        poss.append(pos)
        masks.append(torch.from_numpy(vis).to(dev))
        firsts.append(m)
    at = np.concatenate([[0], np.cumsum(firsts)])
    tok = torch.from_numpy(np.concatenate(seqs)).to(dev)
    x = w["tok_emb"][tok].to(dt) + w["pos_emb"][torch.from_numpy(np.concatenate(poss)).to(dev)].to(dt)
    packed = torch.cat([enc[b, :t] for b, t in enumerate(frames)]).to(dt)
    eat = np.concatenate([[0], np.cumsum(frames)])

    def attend(q, kk, vv, mask):
        q, kk, vv = (t.view(t.shape[0], heads, 64).transpose(0, 1) for t in (q, kk, vv))
        s = q @ kk.transpose(1, 2) / 8.0
        if mask is not None:
            s = s.masked_fill(~mask, -math.inf)
        p = torch.softmax(s, -1)
        return (p @ vv).transpose(0, 1).reshape(-1, d), p

    probs = [None] * B
    for l in range(L):
        y = {n: w["%d.%s" % (l, n)].to(dt) for n, _ in _layer_shapes(d, f)}
        z = _ln(x, y["ln1_g"], y["ln1_b"])
        q, kk, vv = z @ y["wq"].T + y["bq"], z @ y["wk"].T, z @ y["wv"].T + y["bv"]
        a = torch.cat([attend(q[i:j], kk[i:j], vv[i:j], masks[b])[0] for b, (i, j) in enumerate(zip(at, at[1:]))])
        x = x + a @ y["wo"].T + y["bo"]
        q = _ln(x, y["ln2_g"], y["ln2_b"]) @ y["wcq"].T + y["bcq"]
        kk, vv = packed @ y["wck"].T, packed @ y["wcv"].T + y["bcv"]
        a = []
        for b in range(B):
            i, j = eat[b], eat[b + 1]
            o, p = attend(q[at[b]:at[b + 1]], kk[i:j], vv[i:j], None)
            a.append(o)
            if l == _anchor_layer(c):
                probs[b] = p.mean(0)
        x = x + torch.cat(a) @ y["wco"].T + y["bco"]
        z = torch.nn.functional.gelu(_ln(x, y["ln3_g"], y["ln3_b"]) @ y["w1"].T + y["b1"])
        x = x + z @ y["w2"].T + y["b2"]
    rows = torch.cat([torch.arange(at[b] + P0 - 1, at[b + 1]) for b in range(B) if lens[b] >= 0]).to(dev)
    logits = _ln(x[rows], w["lnf_g"], w["lnf_b"]) @ w["tok_emb"].to(dt).T
    best = logits.argmax(-1).cpu().numpy()
    prof = torch.zeros((B, c["frames"]), dtype=dt, device=dev)
    step = np.full((4, B), -1, np.int64)
    path = np.full((B, k), -1, np.int64)
    steps, r0 = [], 0
    for b in range(B):
        step[0, b], step[2, b] = 0, P0 - 1
        if lens[b] < 0:
            continue
        g = best[r0:r0 + firsts[b] - P0 + 1]
        r0 += firsts[b] - P0 + 1
        n = row = 0
        if c["kind"] == "tree":
            while True:
                nxt = [i for i in range(1, lens[b] + 1) if parent[b, i - 1] == row and nodes[b, i - 1] == g[row]]
                if not nxt:
                    break
                row = nxt[0]
                path[b, n] = row
                n += 1
        elif loop:
            n, row = 2 * k + 1, 2 * k + 1
        else:
            while n < lens[b] and block[b, n] == g[n]:
                n += 1
            row = n
        p = probs[b][P0 - 1 + row]
        prof[b, :frames[b]] = p
        step[:, b] = n, g[row], P0 + n, int(p.argmax())
    out = {"profile": prof.cpu()}
    if loop:
        return dict(out, rounds=[None, None])
    out["step"] = step
    if c["kind"] == "tree":
        out["path"] = path
    if c["kind"] == "score":
        out["logits"] = logits.cpu()
    return out
