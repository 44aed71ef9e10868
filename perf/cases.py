"""The measured cases: the calls that a streaming recogniser built on this
framework makes, chunk after chunk.

  greedy   ``Decoder.decode_chunk``, greedy, one n-gram LM, with or without a
           phrase-boosting tree: the framework's main path, from one live
           stream with one-frame chunks to a full server's batch
  lms      the same with several n-gram LMs fused
  pred     the same with the LSTM prediction network (the stateful form)
  beam     ``Decoder.decode_chunk`` with beam search
  encoder  ``Encoder.encode_chunk``: single Conformer blocks and whole encoders

Joint, LSTM and encoder weights, encoder frames and features are drawn from
the seed.  The n-gram LM and the phrase list are the service's fixed
resources: loaded once per process, shared by its decoders.
"""
import functools
import math
import types

import numpy as np
import torch

import paper_2609_14991_gb300 as tsd

DEV = "cuda"
DISCOUNT = 0.7


# ---------------------------------------------------------------- the cases

def _greedy(name, B, V, H, T, order, corpus, phrases, lam, beta, **kw):
    return dict(name=name, kind="greedy", B=B, V=V, H=H, T=T, order=order, corpus=corpus, phrases=phrases, lam=lam,
                beta=beta, max_sym=5, beam=1, n_lm=1, D=0, **kw)


def listed():
    return [
        # one live microphone: the least latency the framework is asked for
        _greedy("greedy one stream", 1, 1024, 640, 13, 4, 600_000, 0, 0.5, 0.0),
        # a few live streams decoded frame by frame (80 ms chunks): the smallest call
        _greedy("greedy 16 frame by frame", 16, 1024, 1024, 1, 6, 1_500_000, 5000, 0.5, 1.5),
        # a small service with a small, odd vocabulary, ragged in every size
        _greedy("greedy 37 odd", 37, 499, 320, 7, 3, 200_000, 16, 0.3, 1.0),
        # the small joint network at the 1040 ms look-ahead
        _greedy("greedy 64", 64, 1024, 640, 13, 4, 600_000, 0, 0.5, 0.0),
        # the large joint network with boosting, an ordinary server's batch
        _greedy("greedy 256", 256, 1024, 1024, 13, 6, 1_500_000, 5000, 0.5, 1.5),
        # a full server: wide vocabulary, long contexts, many phrases (the headline workload)
        _greedy("greedy 1024", 1024, 4096, 1024, 13, 10, 1_200_000, 50000, 0.6, 1.5),
        # a general and a domain LM fused
        dict(_greedy("two lms 256", 256, 1024, 1024, 13, 6, 1_500_000, 5000, 0.5, 1.5), kind="lms", n_lm=2),
        # the prediction network and the joint projections in the loop, at a 400 ms look-ahead
        dict(_greedy("lstm 256", 256, 1024, 1024, 5, 6, 1_500_000, 5000, 0.5, 1.5), kind="pred", D=640),
        # accuracy first: beam search
        dict(_greedy("beam 4 x 128", 128, 1024, 1024, 13, 6, 1_500_000, 5000, 0.5, 1.5), kind="beam", beam=4, max_sym=1),
        # a few live streams through the whole small encoder
        dict(name="encoder 115m x 3", kind="encoder", B=3, C=13, d=512, layers=17, heads=8, ff=2048, warm=0),
        # one block of the large encoder, mid-stream (full left context), an odd batch of short chunks
        dict(name="encoder block 101 x 7", kind="encoder", B=101, C=7, d=1024, layers=1, heads=8, ff=4096, warm=10),
        # a full server's batch through the whole large encoder
        dict(name="encoder 0.6b x 256", kind="encoder", B=256, C=13, d=1024, layers=24, heads=8, ff=4096, warm=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["greedy", "lms", "pred", "beam", "encoder"], [6, 1, 1, 1, 3])[0]
    if kind == "encoder":
        d, heads, ff = rng.choice([(512, 8, 2048), (1024, 8, 4096), (768, 12, 3072), (256, 4, 1024)])
        layers = _log_int(rng, 1, 24)
        return dict(kind="encoder", B=_log_int(rng, 1, 256), C=rng.randint(1, 13), d=d, layers=layers, heads=heads, ff=ff,
                    warm=0 if layers > 4 else rng.randint(0, 6))
    B, V, H, T = _log_int(rng, 1, 1024), _log_int(rng, 256, 4096), 64 * rng.randint(5, 16), rng.randint(1, 13)
    order = rng.randint(3, 8)
    c = dict(kind=kind, B=B, V=V, H=H, T=T, order=order, corpus=_log_int(rng, 150_000, 800_000),
             phrases=rng.choice([0, _log_int(rng, 16, 20000)]), lam=round(rng.uniform(0.3, 0.6), 2),
             beta=round(rng.uniform(0.5, 1.5), 2), max_sym=5, beam=1, n_lm=1, D=0)
    if kind == "lms":
        c.update(n_lm=rng.randint(2, 3), B=min(B, 512))
    elif kind == "pred":
        c.update(D=64 * rng.randint(5, 10), B=min(B, 512), T=rng.randint(1, 5))
    elif kind == "beam":
        c.update(beam=rng.randint(2, 4), B=min(B, 256), V=min(V, 2048), max_sym=1)
    return c


# ------------------------------------------------- the n-gram LM and phrases

class _Lm:
    """A back-off n-gram model estimated from a seeded synthetic corpus by
    absolute discounting.  Windows of one text are closed under prefixes and
    suffixes, as any model estimated from counts is."""

    def __init__(self, V, order, corpus, zipf, seed):
        g = torch.Generator(device=DEV).manual_seed(seed)
        p = torch.arange(1, V + 1, device=DEV, dtype=torch.float64).pow(-zipf).cumsum(0)
        perm = torch.randperm(V, device=DEV, generator=g)
        draw_tok = lambda n: perm[torch.searchsorted(p, torch.rand(n, device=DEV, dtype=torch.float64, generator=g) * p[-1])]
        # half of the text is stock phrases of four labels (so that longer contexts recur), half is fresh
        bank = draw_tok(4 * 20000).view(-1, 4)
        n = corpus // 4
        pick = (torch.rand(n, device=DEV, generator=g).pow(3) * len(bank)).long()
        fresh = torch.rand(n, device=DEV, generator=g) < 0.5
        text = torch.where(fresh[:, None], draw_tok(4 * n).view(-1, 4), bank[pick]).reshape(-1)
        L = len(text)
        ids, n_lo = text, V
        self.V, self.order = V, order
        self.pos, self.tok, self.ctx, self.sfx, self.logp, self.bow = [], [], [], [], [], []
        for k in range(1, order + 1):
            if k == 1:
                cnt = torch.bincount(text, minlength=V).double() + 1
                self.tok.append(torch.arange(V, device=DEV)[:, None])
                self.logp.append((cnt / cnt.sum()).log())
                self.ctx.append(None)
                self.sfx.append(None)
                continue
            lo = ids
            key, ids, c = torch.unique(lo[:L - k + 1] * V + text[k - 1:], sorted=True, return_inverse=True, return_counts=True)
            at = torch.empty(len(key), device=DEV, dtype=torch.long)
            at[ids] = torch.arange(L - k + 1, device=DEV)  # a place where the n-gram stands
            ctx = key // V
            tot = torch.zeros(n_lo, device=DEV, dtype=torch.float64).index_add_(0, ctx, c.double())
            kinds = torch.bincount(ctx, minlength=n_lo).double()
            self.bow.append(torch.where(kinds > 0, (DISCOUNT * kinds / tot.clamp(min=1)).log(), 0.0).nan_to_num(0, 0, 0))
            self.tok.append(text[at[:, None] + torch.arange(k, device=DEV)])
            self.logp.append(((c.double() - DISCOUNT) / tot[ctx]).log())
            self.ctx.append(ctx)
            self.sfx.append(lo[at + 1])  # the n-gram less its first label
            n_lo = len(key)
        self.bow.append(torch.zeros(n_lo, device=DEV, dtype=torch.float64))

    def handle(self):
        f = lambda xs, t: [x.to(t).cpu().numpy() for x in xs]
        return tsd.NGram(self.V, f(self.tok, torch.int32), f(self.logp, torch.float32), f(self.bow, torch.float32))


@functools.lru_cache(maxsize=4)
def _lm_handle(V, order, corpus, zipf, seed):
    return _Lm(V, order, corpus, zipf, seed).handle()


def _lm_args(c, i):
    return c["V"], c["order"], c["corpus"] // (1 + i), 1.05 if c["V"] > 2000 else 1.1, 1000 + i


def _lm_weights(c):
    return [1.0, 0.5, 0.25, 0.25][:c["n_lm"]]


def _phrases(c):
    """c["phrases"] distinct label sequences of 2 to 12 labels, none a prefix of another."""
    r = np.random.RandomState(77)
    n = c["phrases"]
    got = {tuple(r.randint(0, c["V"], r.randint(2, 13))) for _ in range(n)}
    got = sorted(p for p in got if not any(p[:k] in got for k in range(2, len(p))))
    return got


def _boost(c):
    if not c["phrases"]:
        return None
    ph = _phrases(c)
    off = np.cumsum([0] + [len(p) for p in ph]).astype(np.int32)
    return tsd.Boost(c["V"], off, np.concatenate([np.array(p, dtype=np.int32) for p in ph]), 1.0)


@functools.lru_cache(maxsize=4)
def _boost_handle(V, phrases):
    return _boost(dict(V=V, phrases=phrases))


# ------------------------------------------------------------------ decoding

def _randn(g, shape, std):
    return (torch.randn(shape, device=DEV, generator=g) * std).to(torch.bfloat16)


def _decoder_inputs(c, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    V, H, B, T, D = c["V"], c["H"], c["B"], c["T"], c["D"]
    x = types.SimpleNamespace(W=_randn(g, (H, V + 1), 3 / math.sqrt(H)), E=_randn(g, (V + 1, H), 1.0),
                              enc=_randn(g, (B, T, H), 1.0), pred=None)
    if D:
        bias = lambda n: torch.randn(n, device=DEV, generator=g) * 0.1
        bg = bias(4 * D)
        bg[1::4] += 1.0  # the forget gates' usual offset
        x.pred = types.SimpleNamespace(D=D, Henc=H, Ep=_randn(g, (V + 1, D), 1.0), Wg=_randn(g, (2 * D, 4 * D), 1 / math.sqrt(2 * D)),
                                       bg=bg, Wp=_randn(g, (D, H), 3 / math.sqrt(D)), bp=bias(H),
                                       We=_randn(g, (H, H), 1 / math.sqrt(H)), be=bias(H))
    return x


def _bits(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.cpu().numpy()


def _prepare_decoder(c, seed):
    x = _decoder_inputs(c, seed)
    lms = [_lm_handle(*_lm_args(c, i)) for i in range(c["n_lm"])]
    pred = None
    if x.pred:
        pred = types.SimpleNamespace(**{k: v if isinstance(v, int) else _bits(v) for k, v in vars(x.pred).items()})
    how = dict(lms=list(zip(lms, _lm_weights(c)))) if c["n_lm"] > 1 else dict(lm=lms[0])
    boost = _boost_handle(c["V"], c["phrases"]) if c["phrases"] else None
    dec = tsd.Decoder(c["V"], c["H"], x.W, x.E, boost=boost, max_symbols=c["max_sym"], beam_k=c["beam"],
                      max_streams=c["B"], max_T=c["T"], pred=pred, **how)
    out = dec.alloc_out(c["B"], c["T"])
    for t in vars(out).values():
        t.zero_()  # a chunk writes the labels that it emits and leaves the rest
    # an utterance of a beam stream is closed well before its 8192 label-sequence nodes are used up
    utterance = min(128, 8000 // (c["beam"] * c["T"])) if c["beam"] > 1 else None
    return types.SimpleNamespace(c=c, dec=dec, slots=[dec.open() for _ in range(c["B"])], enc=x.enc, out=out,
                                 utterance=utterance, chunks=0)


def _run_decoder(s):
    if s.utterance and s.chunks == s.utterance:
        for slot in s.slots:
            s.dec.close(slot)
        s.slots = [s.dec.open() for _ in s.slots]
        s.chunks = 0
    s.chunks += 1
    s.dec.decode_chunk(s.slots, s.enc, s.c["lam"], s.c["beta"], out=s.out)
    o = s.out
    if s.c["beam"] > 1:
        return {"scores": o.scores, "counts": o.counts}
    return {"tokens": o.tokens, "frames": o.frames, "scores": o.scores, "counts": o.counts}


# ------------------------------------------------------------------- encoder

_LNS = ("ln_ff1", "ln_att", "ln_conv", "ln_ff2", "ln_out")
_FEAT, _STACK, _KERNEL, _LEFT = 80, 8, 9, 70


def _encoder_inputs(c, seed):
    """Weights of one encoder and the chunks of features its streams see: `warm` chunks before the measured one, then that one."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    d, ff = c["d"], c["ff"]
    mat = lambda o, i: _randn(g, (o, i), 1 / math.sqrt(i))
    vec = lambda n, std, mean=0.0: torch.randn(n, device=DEV, generator=g) * std + mean
    layers = []
    for _ in range(c["layers"]):
        L = types.SimpleNamespace(
            ff1_w1=mat(ff, d), ff1_b1=vec(ff, 0.02), ff1_w2=mat(d, ff), ff1_b2=vec(d, 0.02), qkv_w=mat(3 * d, d),
            qkv_b=vec(3 * d, 0.02), pos_w=mat(d, d), pos_u=vec(d, 0.1), pos_v=vec(d, 0.1), out_w=mat(d, d), out_b=vec(d, 0.02),
            pw1_w=mat(2 * d, d), pw1_b=vec(2 * d, 0.02), dw_w=vec((d, _KERNEL), 1 / math.sqrt(_KERNEL)), dw_b=vec(d, 0.02),
            bn_scale=vec(d, 0.1, 1.0), bn_shift=vec(d, 0.05), pw2_w=mat(d, d), pw2_b=vec(d, 0.02), ff2_w1=mat(ff, d),
            ff2_b1=vec(ff, 0.02), ff2_w2=mat(d, ff), ff2_b2=vec(d, 0.02))
        for n in _LNS:
            setattr(L, n, (vec(d, 0.1, 1.0), vec(d, 0.05)))
        layers.append(L)
    w = types.SimpleNamespace(sub_w=mat(d, _STACK * _FEAT), sub_b=vec(d, 0.02), layers=layers)
    chunks = [_randn(g, (c["B"], c["C"] * _STACK, _FEAT), 1.0) for _ in range(c["warm"] + 1)]
    return w, chunks


def _prepare_encoder(c, seed):
    w, chunks = _encoder_inputs(c, seed)
    host = lambda v: tuple(_bits(x) for x in v) if isinstance(v, tuple) else _bits(v)
    hw = types.SimpleNamespace(
        cfg=types.SimpleNamespace(d=c["d"], heads=c["heads"], ff=c["ff"], kernel=_KERNEL, left=_LEFT, chunk=c["C"], feat=_FEAT,
                                  stack=_STACK),
        sub_w=host(w.sub_w), sub_b=host(w.sub_b),
        layers=[types.SimpleNamespace(**{k: host(v) for k, v in vars(L).items()}) for L in w.layers])
    enc = tsd.Encoder(hw, max_streams=c["B"])
    slots = [enc.open() for _ in range(c["B"])]
    for x in chunks[:-1]:
        enc.encode_chunk(slots, x)
    return types.SimpleNamespace(c=c, enc=enc, slots=slots, feats=chunks[-1])


def _run_encoder(s):
    return s.enc.encode_chunk(s.slots, s.feats).view(torch.bfloat16)


# -------------------------------------------------------------- the interface

def prepare(case, seed):
    return _prepare_encoder(case, seed) if case["kind"] == "encoder" else _prepare_decoder(case, seed)


def run(state):
    return _run_encoder(state) if state.c["kind"] == "encoder" else _run_decoder(state)


def work(case):
    c = case
    if c["kind"] == "encoder":
        M, d, ff, n = c["B"] * c["C"], c["d"], c["ff"], c["layers"]
        per = 4 * d * ff + 7 * d * d  # weights of a block's matrices
        left = min(_LEFT, _LEFT if c["warm"] else c["C"])
        cache = c["B"] * n * (left * 2 * d + (_KERNEL - 1) * d) * 2  # keys, values and convolution frames read
        new = c["B"] * n * (min(c["C"], _LEFT) * 2 * d + (_KERNEL - 1) * d) * 2  # and written
        attn = 2 * c["B"] * c["C"] * n * d * (2 * (left + c["C"]) + (left + 2 * c["C"]))
        return {"flops": 2 * M * (n * per + _STACK * _FEAT * d) + attn,
                "bytes": 2 * (n * per + _STACK * _FEAT * d) + 2 * M * (_STACK * _FEAT + d) + cache + new}
    rows, steps, N = c["B"] * c["beam"], c["T"] * c["max_sym"], c["V"] + 1
    # each row-step reads the LM's continuations of its state (about an eighth of the labels, 8 bytes each)
    b = 2 * N * c["H"] * 2 + 2 * c["B"] * c["T"] * c["H"] + rows * steps * c["n_lm"] * N + 12 * c["B"] * steps
    f = 2 * rows * steps * c["H"] * N
    if c["D"]:
        D, H = c["D"], c["H"]
        b += 2 * (8 * D * D + D * H + H * H + N * D)
        f += 2 * rows * (steps * (8 * D * D + D * H) + c["T"] * H * H)
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "encoder":
        # a matrix product's operands are bf16: a sum taken in another order rounds some of them the other way, and
        # that travels on.  Seen with every such rounding left out: 0.0023 after one block, 0.0057 after 24.
        return {"rel": min(0.02, 0.008 + 0.0006 * case["layers"]), "max": 0.12}
    if case["kind"] == "pred":
        # the LSTM's output is kept in bf16 and fed back: a rounding the other way can divert a stream for the rest
        # of the chunk.  Seen against 64 bits: up to 0.04 over five frames, so the most that can be stated.
        return {"rel": 0.03, "max": 0.9, "differ": 0.01}
    # scores are 3e-7 off where no label changes.  Once in some ten thousand label steps the two best labels are
    # as near as 32-bit sums can tell, and a stream that takes the other one differs for the rest of its chunk: seen
    # as 3.6e-4 in one of nine decodes.
    return {"rel": 1.5e-3, "max": 0.9, "differ": 0.002}


# ------------------------------------------------- the same in 64-bit floats

class _Tree:
    """A tree of label sequences with suffix links, shared by the LM and the
    phrases: node -> its continuations (sorted by label) and its suffix."""

    def __init__(self, V, begin, count, tok, to, sfx):
        self.V, self.begin, self.count, self.tok, self.to, self.sfx = V, begin, count, tok, to, sfx
        node = torch.repeat_interleave(torch.arange(len(begin), device=DEV), count)
        self.key = node * V + tok  # ascending: continuations are grouped by node

    def spread(self, cur):
        """(row, continuation) of every continuation of the rows' nodes."""
        n = self.count[cur]
        row = torch.repeat_interleave(torch.arange(len(cur), device=DEV), n)
        first = torch.cumsum(n, 0) - n
        return row, self.begin[cur][row] + torch.arange(len(row), device=DEV) - first[row]

    def find(self, cur, y):
        """The continuation y of each node, or -1."""
        k = cur * self.V + y
        i = torch.searchsorted(self.key, k).clamp(max=len(self.key) - 1)
        return torch.where(self.key[i] == k, i, -1)


class _ExactLm(_Tree):
    def __init__(self, lm):
        n = [len(x) for x in lm.logp]
        base = np.cumsum([1] + n)  # node 0 is the empty context
        self.uni = lm.logp[0]
        S = int(base[lm.order - 1])
        begin, count = (torch.zeros(S, device=DEV, dtype=torch.long) for _ in range(2))
        sfx = torch.zeros(S, device=DEV, dtype=torch.long)
        self.bow = torch.zeros(S, device=DEV, dtype=torch.float64)
        tok, to, logp, off = [], [], [], 0
        for k in range(2, lm.order + 1):
            a, m = int(base[k - 2]), n[k - 2]
            count[a:a + m] = torch.bincount(lm.ctx[k - 1], minlength=m)
            begin[a:a + m] = off + torch.cumsum(count[a:a + m], 0) - count[a:a + m]
            self.bow[a:a + m] = lm.bow[k - 2]
            if k > 2:
                sfx[a:a + m] = int(base[k - 3]) + lm.sfx[k - 2]
            tok.append(lm.tok[k - 1][:, -1])
            logp.append(lm.logp[k - 1])
            to.append(torch.arange(n[k - 1], device=DEV) + int(base[k - 1]) if k < lm.order else torch.full((n[k - 1],), -1, device=DEV))
            off += n[k - 1]
        # the inputs are 32-bit: what the model is
        self.uni, self.bow, self.logp = self.uni.float().double(), self.bow.float().double(), torch.cat(logp).float().double()
        super().__init__(lm.V, begin, count, torch.cat(tok), torch.cat(to), sfx)

    def rows(self, state):
        """log p(v | state) for every label."""
        out = torch.full((len(state), self.V), math.nan, device=DEV, dtype=torch.float64)
        off = torch.zeros(len(state), device=DEV, dtype=torch.float64)
        cur = state
        while bool((cur > 0).any()):
            row, i = self.spread(cur)
            m = out[row, self.tok[i]].isnan()
            row, i = row[m], i[m]
            out[row, self.tok[i]] = off[row] + self.logp[i]
            off = off + self.bow[cur]
            cur = self.sfx[cur]
        return torch.where(out.isnan(), self.uni + off[:, None], out)

    def step(self, state, y):
        new, cur = torch.zeros_like(state), state
        while True:
            i = torch.where(cur > 0, self.find(cur, y), -1)
            t = torch.where(i >= 0, self.to[i.clamp(min=0)], -1)
            new = torch.where((new == 0) & (t > 0), t, new)
            if not bool((cur > 0).any()):
                return torch.where(new == 0, 1 + y, new)
            cur = self.sfx[cur]


class _ExactBoost(_Tree):
    def __init__(self, V, phrases):
        kids, ends = [{}], set()
        parent, label = [0], [0]
        for p in phrases:
            q = 0
            for t in p:
                if t not in kids[q]:
                    kids[q][t] = len(kids)
                    kids.append({})
                    parent.append(q)
                    label.append(int(t))
                q = kids[q][t]
            ends.add(q)
        fail, depth = [0] * len(kids), [0] * len(kids)
        order = [0]
        for q in order:
            order.extend(kids[q].values())
        for q in order[1:]:
            depth[q] = depth[parent[q]] + 1
            f = parent[q]
            while f and label[q] not in kids[fail[f]]:
                f = fail[f]
            fail[q] = kids[fail[f]].get(label[q], 0) if f else 0
        items = [sorted(k.items()) for k in kids]
        T = lambda v: torch.tensor(v, device=DEV, dtype=torch.long)
        count = T([len(i) for i in items])
        super().__init__(V, torch.cumsum(count, 0) - count, count, T([t for i in items for t, _ in i]),
                         T([q for i in items for _, q in i]), T(fail))
        self.depth, self.end = T(depth), torch.tensor([q in ends for q in range(len(kids))], device=DEV)

    def rows(self, node):
        """Depth of the longest match after each label, less the present one."""
        out = torch.full((len(node), self.V), -1, device=DEV, dtype=torch.long)
        cur = node
        while True:
            row, i = self.spread(cur)
            m = out[row, self.tok[i]] < 0
            row, i = row[m], i[m]
            out[row, self.tok[i]] = self.depth[self.to[i]]
            if not bool((cur > 0).any()):
                break
            cur = self.sfx[cur]
        return (out.clamp(min=0) - self.depth[node][:, None]).double()

    def step(self, node, y):
        new, cur = torch.zeros_like(node), node
        while True:
            i = self.find(cur, y)
            new = torch.where((new == 0) & (i >= 0), self.to[i.clamp(min=0)], new)
            if not bool((cur > 0).any()):
                return torch.where(self.end[new], 0, new)
            cur = self.sfx[cur]


def _bf16(x):
    return x.float().to(torch.bfloat16).double()


class _ExactDecoder:
    def __init__(self, c, seed):
        self.c, self.x = c, _decoder_inputs(c, seed)
        self.W = self.x.W.double()
        self.lms = [(_ExactLm(_Lm(*_lm_args(c, i))), w) for i, w in enumerate(_lm_weights(c))]
        self.boost = _ExactBoost(c["V"], _phrases(c)) if c["phrases"] else None

    def fused(self, A, states, node):
        """Eq. 1 over the V labels and blank for rows of joint input."""
        c = self.c
        s = torch.log_softmax(A @ self.W, 1)
        for (lm, w), st in zip(self.lms, states):
            s[:, :-1] += c["lam"] * w * lm.rows(st)
        if self.boost is not None:
            s[:, :-1] += c["beta"] * self.boost.rows(node)
        return s

    def step(self, states, node, y):
        return [lm.step(st, y) for (lm, _), st in zip(self.lms, states)], self.boost.step(node, y) if self.boost is not None else node


def _exact_greedy(c, seed):
    e = _ExactDecoder(c, seed)
    B, T, V, S = c["B"], c["T"], c["V"], c["max_sym"]
    zero = lambda: torch.zeros(B, device=DEV, dtype=torch.long)
    t, sym, cnt, last, node = zero(), zero(), zero(), zero() + V, zero()
    states = [zero() for _ in e.lms]
    scores = torch.zeros(B, T * S, device=DEV, dtype=torch.float64)
    p = e.x.pred
    if p is not None:
        Ep, Wg, Wp = p.Ep.double(), p.Wg.double(), p.Wp.double()
        penc = e.x.enc.double() @ p.We.double() + p.be.double()

        def cell(y, h, cc):
            g = (torch.cat([Ep[y], h], 1) @ Wg + p.bg.double()).view(B, -1, 4)
            cc = g[..., 1].sigmoid() * cc + g[..., 0].sigmoid() * g[..., 2].tanh()
            return _bf16(g[..., 3].sigmoid() * cc.tanh()), cc

        h, cc = cell(last, *(torch.zeros(B, c["D"], device=DEV, dtype=torch.float64) for _ in range(2)))
    rows = torch.arange(B, device=DEV)
    for _ in range(T * S):
        on = t < T
        at = t.clamp(max=T - 1)
        if p is None:
            A = torch.relu(e.x.enc[rows, at].float() + e.x.E[last].float()).to(torch.bfloat16).double()
        else:
            A = _bf16(torch.relu(penc[rows, at] + h @ Wp + p.bp.double()))
        best, y = e.fused(A, states, node).max(1)
        emit = on & (y < V)
        scores[rows[emit], cnt[emit]] = best[emit]
        yc = y.clamp(max=V - 1)
        st2, nd2 = e.step(states, node, yc)
        states = [torch.where(emit, a, b) for a, b in zip(st2, states)]
        node = torch.where(emit, nd2, node)
        last = torch.where(emit, y, last)
        if p is not None:
            h2, c2 = cell(yc, h, cc)
            h, cc = torch.where(emit[:, None], h2, h), torch.where(emit[:, None], c2, cc)
        cnt, sym = cnt + emit, sym + emit.long()
        go = on & (~emit | (sym >= S))
        t, sym = t + go, torch.where(go, 0, sym)
    return {"tokens": None, "frames": None, "scores": scores, "counts": None}


def _exact_beam(c, seed):
    e = _ExactDecoder(c, seed)
    B, T, V, K = c["B"], c["T"], c["V"], c["beam"]
    # per stream a list of (score, labels, LM states, trie node)
    beams = [[(0.0, (), [0] * len(e.lms), 0)] for _ in range(B)]
    L = lambda v: torch.tensor(v, device=DEV, dtype=torch.long)
    for t in range(T):
        flat = [(b, h) for b in range(B) for h in beams[b]]
        own = L([b for b, _ in flat])
        last = L([h[1][-1] if h[1] else V for _, h in flat])
        A = torch.relu(e.x.enc[own, t].float() + e.x.E[last].float()).to(torch.bfloat16).double()
        states, node = [L([h[2][i] for _, h in flat]) for i in range(len(e.lms))], L([h[3] for _, h in flat])
        total = e.fused(A, states, node) + torch.tensor([h[0] for _, h in flat], device=DEV, dtype=torch.float64)[:, None]
        val, lab = total.topk(K, 1)  # a stream keeps K extensions in all, so at most K of one hypothesis
        cand = [[] for _ in range(B)]
        for j, (b, h) in enumerate(flat):
            cand[b].append(j)
        val, lab = val.cpu().numpy(), lab.cpu().numpy()
        kept = []
        for b in range(B):
            ext = sorted((-val[j, k], j, int(lab[j, k])) for j in cand[b] for k in range(K))[:K]
            kept.append([(-v, j, y) for v, j, y in ext])
        src, ys = L([j for k in kept for _, j, _ in k]), L([min(y, V - 1) for k in kept for _, _, y in k])
        st2, nd2 = e.step([s[src] for s in states], node[src], ys)
        st2, nd2 = [s.tolist() for s in st2], nd2.tolist()
        i = 0
        for b in range(B):
            new = {}
            for v, j, y in kept[b]:
                _, labels, st, nd = flat[j][1]
                if y < V:
                    labels, st, nd = labels + (y,), [s[i] for s in st2], nd2[i]
                i += 1
                if labels in new:
                    new[labels][0] = float(np.logaddexp(new[labels][0], v))
                else:
                    new[labels] = [v, labels, st, nd]
            beams[b] = [tuple(h) for h in new.values()]
    scores = torch.zeros(B, T * c["max_sym"], device=DEV, dtype=torch.float64)
    scores[:, 0] = torch.tensor([max(h[0] for h in hs) for hs in beams], device=DEV, dtype=torch.float64)
    return {"scores": scores, "counts": None}


def _exact_encoder(c, seed):
    w, chunks = _encoder_inputs(c, seed)
    B, C, d, nh = c["B"], c["C"], c["d"], c["heads"]
    dh = d // nh
    ln = lambda x, gb: torch.nn.functional.layer_norm(x, (d,), gb[0].double(), gb[1].double(), 1e-5)
    lin = lambda x, m, b: x @ m.double().t() + b.double()
    swish = lambda x: x * x.sigmoid()
    half = torch.arange(d, device=DEV, dtype=torch.float64) // 2
    freq = 10000.0 ** (-2 * half / d)
    kv = [None] * c["layers"]
    cv = [torch.zeros(B, _KERNEL - 1, d, device=DEV, dtype=torch.float64) for _ in w.layers]
    for f in chunks:
        x = lin(f.double().view(B, C, -1), w.sub_w, w.sub_b)
        for l, L in enumerate(w.layers):
            x = x + 0.5 * lin(swish(lin(ln(x, L.ln_ff1), L.ff1_w1, L.ff1_b1)), L.ff1_w2, L.ff1_b2)
            q, k, v = lin(ln(x, L.ln_att), L.qkv_w, L.qkv_b).split(d, -1)
            if kv[l] is not None:
                k, v = torch.cat([kv[l][0], k], 1), torch.cat([kv[l][1], v], 1)
            W = k.shape[1]
            delta = (W - C + torch.arange(C, device=DEV))[:, None] - torch.arange(W, device=DEV)
            r = delta[..., None] * freq
            r = torch.where(torch.arange(d, device=DEV) % 2 == 1, r.cos(), r.sin())
            P = (r @ L.pos_w.double().t()).view(C, W, nh, dh)
            qh, kh, vh = (z.view(B, -1, nh, dh) for z in (q, k, v))
            s = torch.einsum("bihe,bjhe->bhij", qh + L.pos_u.double().view(nh, dh), kh)
            s = s + torch.einsum("bihe,ijhe->bhij", qh + L.pos_v.double().view(nh, dh), P)
            a = torch.einsum("bhij,bjhe->bihe", (s / math.sqrt(dh)).softmax(-1), vh).reshape(B, C, d)
            x = x + lin(a, L.out_w, L.out_b)
            kv[l] = (k[:, -_LEFT:], v[:, -_LEFT:])
            a, g = lin(ln(x, L.ln_conv), L.pw1_w, L.pw1_b).split(d, -1)
            seq = torch.cat([cv[l], a * g.sigmoid()], 1)
            cv[l] = seq[:, -(_KERNEL - 1):]
            y = torch.nn.functional.conv1d(seq.transpose(1, 2), L.dw_w.double()[:, None], groups=d).transpose(1, 2) + L.dw_b.double()
            x = x + lin(swish(y * L.bn_scale.double() + L.bn_shift.double()), L.pw2_w, L.pw2_b)
            x = x + 0.5 * lin(swish(lin(ln(x, L.ln_ff2), L.ff2_w1, L.ff2_b1)), L.ff2_w2, L.ff2_b2)
            x = ln(x, L.ln_out)
    return x


def exact(case, seed):
    if case["kind"] == "encoder":
        return _exact_encoder(case, seed)
    return _exact_beam(case, seed) if case["kind"] == "beam" else _exact_greedy(case, seed)
