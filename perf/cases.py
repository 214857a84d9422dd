"""Workloads of the speculative-decoding library, each through its public entry points.

A case is a dict of plain values.  Its "kind" says which call of a serving program it stands for:

  verify       ssd_verify + ssd_kv_commit, the step of Algorithm 1 that the target model runs
  verify_host  the same from and to pinned host buffers
  draft        one ssd_draft_step
  iteration    several ssd_iteration calls: what a streaming synthesizer emits as one chunk
  prefill      a prompt enters the cache

Model shapes are those of the repository's five configurations.  Every pass starts from the same
prefix: the rollback that puts the streams back there (ssd_kv_restore) is part of the pass.
"""
import functools
import math

import numpy as np
import torch

from paper_2505_15380_b200 import binding, synth

DEVICE = "cuda:0"
ROOM = 256  # tokens a stream may still emit: its cache is made for the whole utterance

SHAPES = {
    "tiny": synth.workload(0).target,    # 2 layers, fp32
    "half_b": synth.workload(1).target,  # 24 layers, d 896: the paper's target
    "large": synth.workload(4).target,   # 28 layers, d 1536
    "small": synth.workload(1).draft,    # 4 layers, d 512
}
INHERITED_LAYERS = tuple(range(0, 24, 3))  # the paper's draft: 8 of the target's 24 layers


# ------------------------------------------------------------------------------------- cases

def _case(kind, model, batch, gamma, lo, hi, **more):
    c = {"kind": kind, "model": model, "batch": batch, "gamma": gamma, "prefix_lo": lo, "prefix_hi": hi,
         "temperature": 1.0, "top_k": 0, "top_p": 0.0, "ras_window": 0, "beta": 0.4, "paged": False,
         "draft": "", "iterations": 0, "n_in": 0}
    c.update(more)
    return c


def listed():
    return [
        # configuration 0: the fp32 model, smallest call of all
        dict(_case("verify", "tiny", 1, 4, 64, 64), name="verify_fp32_tiny"),
        # one draft step of one stream as a host-driven loop makes it
        dict(_case("draft", "small", 1, 0, 301, 301, n_in=1), name="draft_step_b1"),
        # configuration 1: one utterance, a 3 s voice prompt and the text before it
        dict(_case("verify", "half_b", 1, 4, 300, 300), name="verify_b1_g4_n300"),
        # the same for a program that keeps its data on the host
        dict(_case("verify_host", "half_b", 1, 4, 300, 300), name="verify_host_b1_g4_n300"),
        # configuration 2's far corner: the longest draft over a long prefix, an odd row count
        dict(_case("verify", "half_b", 1, 8, 1999, 1999), name="verify_b1_g8_n1999"),
        # a few utterances on a paged cache with the CosyVoice sampler (nucleus + repetition-aware)
        dict(_case("verify", "half_b", 6, 3, 150, 900, paged=True, temperature=1.0, top_k=25, top_p=0.8,
                   ras_window=10), name="verify_paged_b6_g3"),
        # configuration 3: a batch of ragged utterances
        dict(_case("verify", "half_b", 16, 5, 200, 1500, temperature=0.8, top_k=25), name="verify_b16_g5_ragged"),
        # configuration 4: the large model, a full server
        dict(_case("verify", "large", 64, 6, 4096, 4096, temperature=0.8, top_k=25), name="verify_large_b64_g6"),
        # the whole of Algorithm 1 on the device with a small draft
        dict(_case("iteration", "half_b", 1, 4, 300, 300, draft="small", iterations=8), name="iterate_b1_g4"),
        # the paper's own setting (gamma 3, a draft made of 8 target layers), a few streams
        dict(_case("iteration", "half_b", 3, 3, 200, 700, draft="inherited", iterations=4, top_p=0.8, ras_window=10),
             name="iterate_b3_g3_inherited"),
        # a new utterance: text and voice prompt
        dict(_case("prefill", "half_b", 1, 4, 301, 301), name="prefill_b1_n301"),
        # utterances with long context join together
        dict(_case("prefill", "half_b", 8, 5, 200, 1500), name="prefill_b8_ragged"),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


_SAMPLERS = ({}, {"temperature": 0.8, "top_k": 25}, {"top_p": 0.8}, {"top_k": 25, "top_p": 0.8, "ras_window": 10})


def draw(rng):
    kind = rng.choice(("verify", "verify", "verify", "verify_large", "verify_host", "draft", "iteration", "prefill",
                       "verify_tiny"))
    s = dict(rng.choice(_SAMPLERS), beta=rng.choice((0.0, 0.2, 0.4)))
    if kind == "verify_tiny":
        return _case("verify", "tiny", rng.randint(1, 4), rng.randint(1, 8), n := _log(rng, 16, 512), n, **s)
    if kind == "verify_large":
        n = _log(rng, 256, 4096)
        return _case("verify", "large", _log(rng, 1, 64), rng.randint(1, 6), n, n, **s)
    if kind == "draft":
        n = _log(rng, 16, 2048)
        model = rng.choice(("small", "half_b"))
        return _case("draft", model, rng.randint(1, 8), 0, n, n, n_in=rng.randint(1, 2), **s)
    if kind == "prefill":
        n = _log(rng, 20, 1500)
        return _case("prefill", "half_b", rng.randint(1, 8), rng.randint(2, 8), max(2, n // rng.randint(1, 4)), n)
    lo = _log(rng, 16, 1800)
    hi = rng.randint(lo, min(2 * lo, 2048))
    if kind == "iteration":
        g = rng.randint(2, 6)
        return _case("iteration", "half_b", rng.randint(1, 4), g, lo, hi, draft=rng.choice(("small", "inherited")),
                     iterations=4, **s)
    return _case(kind, "half_b", _log(rng, 1, 32), rng.randint(1, 8), lo, hi,
                 paged=kind == "verify" and rng.random() < 0.3, **s)


def _lengths(case):
    return synth.ragged_lengths(case["batch"], case["prefix_lo"], case["prefix_hi"], 3)


# ------------------------------------------------------------------------------------- models

@functools.lru_cache(maxsize=None)
def _model(name):
    """Random-init weights of a shape, N(0, 0.02) with unit gains; a server loads them once."""
    if name == "inherited":
        return binding.InheritedModel(_model("half_b"), INHERITED_LAYERS)
    shape = SHAPES[name]
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(1000 + sorted(SHAPES).index(name))
    fp32 = shape.weight_dtype == synth.F32
    parts = []
    for tensor, dims in shape.tensor_list():
        n = int(np.prod(dims))
        w = (torch.ones(n, device=DEVICE) if "norm" in tensor else
             torch.randn(n, generator=gen, device=DEVICE) * 0.02)
        w = w.cpu() if fp32 else w.to(torch.bfloat16).view(torch.int16).cpu()
        parts.append(w.numpy())
    blob = np.concatenate(parts)
    return binding.Model(shape, blob if fp32 else blob.view(np.uint16), device=DEVICE)


# ------------------------------------------------------------------------------------- states

def _prefix_ids(shape, n, seed, stream):
    """Text ids (a fifth of the prompt, up to 60), then speech ids; the last one is pending."""
    rng = np.random.Generator(np.random.Philox(key=[seed, 1 + stream]))
    ids = rng.integers(0, shape.vocab_out, size=n).astype(np.int32)
    nt = min(60, n // 5) if shape.vocab_text else 0
    ids[:nt] = shape.vocab_out + rng.integers(0, shape.vocab_text, size=nt) if nt else ids[:nt]
    return ids


def _streams(case, model, lens, max_gamma, seed):
    """Streams that hold seeded prefixes of lens[b] - 1 cached tokens and one pending token."""
    cap = max(lens) + ROOM
    prefixes = [_prefix_ids(model.shape, n, seed, b) for b, n in enumerate(lens)]
    cached, pending = [n - 1 for n in lens], [int(p[-1]) for p in prefixes]
    B = len(lens)
    if case["paged"]:
        per = -(-cap // binding.PagedStreams.PAGE_TOKENS)
        st = binding.PagedStreams(model, B, B * per, per, max_gamma)
        st.kv.zero_()
        st.kv_truncate(cached, pending)
        st.forward(torch.zeros((B, 1), dtype=torch.int32, device=DEVICE), 1,    # the prefixes get their pages
                   torch.empty((B, 2, model.shape.vocab_out), device=DEVICE))
        gen = torch.Generator(device=DEVICE)
        gen.manual_seed(seed)
        _, _, table = st.paged_state()
        for b in range(B):
            pages = torch.from_numpy(table[b, : -(-cached[b] // 64)].astype(np.int64)).to(DEVICE)
            if len(pages):
                shape = (st.kv.shape[0], len(pages)) + tuple(st.kv.shape[2:])
                st.kv[:, pages] = (torch.randn(shape, generator=gen, device=DEVICE) * 0.6).to(st.kv.dtype)
    else:
        st = binding.Streams(model, B, cap, max_gamma)
        st.kv.zero_()
        synth.fill_synthetic_kv(st.kv, cached, seed=seed)
    st.kv_truncate(cached, pending)
    return st, prefixes


def _start(lens, prefixes, back=1):
    """Device copies of the state to roll back to."""
    return (torch.tensor([n - back for n in lens], dtype=torch.int32, device=DEVICE),
            torch.tensor([int(p[-1]) for p in prefixes], dtype=torch.int32, device=DEVICE))


def _rows(st, lens, first, count):
    """Views of the cache slots lens[b] + first .. + count of every stream."""
    if len(set(lens)) == 1:
        return [st.kv[:, :, :, :, lens[0] + first: lens[0] + first + count]]
    return [st.kv[:, b, :, :, n + first: n + first + count] for b, n in enumerate(lens)]


def _draft_rows(case, shape, gen):
    """What a draft model hands over: rows p over the sampler's support and tokens drawn from them."""
    B, g, V = case["batch"], case["gamma"], shape.vocab_out
    z = torch.randn((B, g, V), generator=gen, device=DEVICE) * (0.6 / case["temperature"])
    if case["top_k"]:
        kth = torch.topk(z, case["top_k"], dim=-1).values[..., -1:]
        z = torch.where(z >= kth, z, torch.full_like(z, -math.inf))
    p = torch.softmax(z, dim=-1)
    x = torch.multinomial(p.view(B * g, V), 1, generator=gen).view(B, g).to(torch.int32)
    return x.contiguous(), p.contiguous()


def _params(case, recent=None):
    return binding.VerifyParams(case["gamma"], case["temperature"], case["top_k"], case["beta"], case["top_p"],
                                case["ras_window"], 0.1 if case["ras_window"] else 0.0,
                                recent.data_ptr() if recent is not None else None)


def _recent(case, prefixes):
    w = case["ras_window"]
    if not w:
        return None
    rec = np.full((len(prefixes), w), -1, dtype=np.int32)
    for b, p in enumerate(prefixes):
        tail = p[-w:]
        rec[b, w - len(tail):] = tail
    return torch.from_numpy(rec).to(DEVICE)


def prepare(case, seed):
    model = _model(case["model"])
    shape, B, g = model.shape, case["batch"], case["gamma"]
    lens = _lengths(case)
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed + 1)
    s = {"case": case}
    if case["kind"] == "prefill":
        st = binding.Streams(model, B, max(lens) + ROOM, g)
        st.kv.zero_()
        prefixes = [_prefix_ids(shape, n, seed, b) for b, n in enumerate(lens)]
        s.update(st=st, prefixes=prefixes, start=_start([0] * B, prefixes, 0),
                 kv=[st.kv[:, b, :, :, : n - 1] for b, n in enumerate(lens)])
        return s
    st, prefixes = _streams(case, model, lens, max(g, 1), seed)
    s.update(st=st, start=_start(lens, prefixes))
    if case["kind"] == "draft":
        n = case["n_in"]
        s.update(ids=torch.from_numpy(np.stack([p[-2:][-n:] for p in prefixes])).to(DEVICE).contiguous(),
                 start=_start(lens, prefixes, n), par=binding.VerifyParams(
                     1, case["temperature"], case["top_k"], 0.0, case["top_p"], 0, 0.0, None),
                 uni=torch.from_numpy(synth.verify_uniforms(seed, B, 1)[:, 0, 0].copy()).to(DEVICE),
                 token=torch.zeros(B, dtype=torch.int32, device=DEVICE),
                 row=torch.zeros((B, shape.vocab_out), device=DEVICE), kv=_rows(st, lens, -n, n))
        return s
    if case["kind"] == "iteration":
        it, per = case["iterations"], g + 2 * (g + 1)
        ds, _ = _streams(case, _model(case["draft"]), lens, g, seed)
        pool = np.stack([synth.verify_uniforms(seed, B, per, step=i)[:, :, 0] for i in range(it)])
        loop = binding.Loop(st, ds, prefixes, g, pool.astype(np.float32), it * (g + 1),
                            ras_window=case["ras_window"])
        s.update(ds=ds, loop=loop, par=_params(case, loop.recent), ids=loop.in_ids.clone(),
                 recent=loop.recent.clone() if loop.recent is not None else None,
                 dstart=_start(lens, prefixes, 2), kv=_rows(st, lens, -1, it * (g + 1)))
        return s
    x, p = _draft_rows(case, shape, gen)
    u = torch.from_numpy(synth.verify_uniforms(seed, B, g + 1)).to(DEVICE)
    k, y = (torch.zeros(B, dtype=torch.int32, device=DEVICE) for _ in range(2))
    s["recent"] = _recent(case, prefixes)
    s["par"] = _params(case, s["recent"])
    s["kv"] = [] if case["paged"] else _rows(st, lens, -1, g + 1)
    if case["kind"] == "verify_host":
        x, p, u, k, y = (t.cpu().pin_memory() for t in (x, p, u, k, y))
    else:
        s["logits"] = torch.zeros((B, g + 1, shape.vocab_out), device=DEVICE)
    s.update(x=x, p=p, u=u, k=k, y=y)
    return s


# ------------------------------------------------------------------------------------- a pass

def run(s):
    kind, st = s["case"]["kind"], s["st"]
    st.kv_restore(*s["start"])
    if kind == "prefill":
        st.prefill(s["prefixes"])
        return s["kv"]
    if kind == "draft":
        st.draft_step(s["ids"], s["case"]["n_in"], s["uni"], s["par"], s["token"], s["row"])
        return [s["token"], s["row"]] + s["kv"]
    if kind == "iteration":
        loop = s["loop"]
        s["ds"].kv_restore(*s["dstart"])
        loop.iteration.zero_()
        loop.out_count.zero_()
        loop.in_ids.copy_(s["ids"])
        if s["recent"] is not None:
            loop.recent.copy_(s["recent"])
        for _ in range(s["case"]["iterations"]):
            loop.iterate(s["par"])
        return [loop.out_tokens, loop.out_count, loop.accept_log, loop.draft_tokens, loop.draft_probs] + s["kv"]
    if kind == "verify_host":
        st.verify_host(s["x"], s["p"], s["u"], s["par"], s["k"], s["y"])
        return [s["k"], s["y"]] + s["kv"]
    st.verify(s["x"], s["p"], s["u"], s["par"], s["k"], s["y"], s["logits"])
    st.kv_commit(s["k"], s["y"])
    return [s["k"], s["y"], s["logits"]] + s["kv"]


# ------------------------------------------------------------------------------------- yardsticks

def _forward_work(shape, lens, rows, head):
    """Bytes and operations of one decoder forward of `rows` rows per stream over lens[b] cached tokens."""
    el = 4 if shape.weight_dtype == synth.F32 else 2
    head_el = shape.vocab_out * shape.d_model
    w = shape.streamed_weight_bytes() - (0 if head else head_el * el)
    M = len(lens) * rows
    flops = 2.0 * (w / el - (head_el if head else 0)) * M + (2.0 * head_el * M if head else 0)
    flops += sum(4.0 * shape.n_layers * shape.q_dim * rows * (n + (rows + 1) / 2) for n in lens)
    return w + shape.kv_bytes_per_token() * sum(n + rows for n in lens), flops


def work(case):
    shape, lens, g = SHAPES[case["model"]], _lengths(case), case["gamma"]
    B, V = case["batch"], shape.vocab_out
    if case["kind"] == "prefill":  # one pass over the weights, every row computed and cached once
        w, _ = _forward_work(shape, [], 1, False)
        flops = sum(_forward_work(shape, [0], n - 1, False)[1] for n in lens)
        return {"bytes": w + shape.kv_bytes_per_token() * sum(n - 1 for n in lens), "flops": flops}
    if case["kind"] == "draft":
        n = case["n_in"]
        by, fl = _forward_work(shape, [v - n for v in lens], n, True)
        return {"bytes": by + B * V * 4, "flops": fl}
    by, fl = _forward_work(shape, [n - 1 for n in lens], g + 1, True)
    by += B * g * V * 4 + (B * (g + 1) * V * 4 if case["kind"] == "verify" else 0)
    if case["kind"] == "iteration":
        d = SHAPES["small"] if case["draft"] == "small" else _model("inherited").shape
        for i in range(g):
            b1, f1 = _forward_work(d, [n - 2 + (i and i + 1) for n in lens], 1 if i else 2, True)
            by, fl = by + b1 + B * V * 4, fl + f1
        by, fl = by * case["iterations"], fl * case["iterations"]
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Whole numbers stay; fp32 sums to 1e-5.  Cached keys and values are bf16: sums taken in another
    order move a few of them by one step (2**-8), and the later layers and the logits with them."""
    if case["model"] == "tiny":
        return {"rel": 2e-5, "max": 2e-4}
    return {"rel": 1e-3, "max": 3e-2}
