"""The work this library is given by a program that decodes under a grammar, as cases that can be timed.

Every case goes through the public entry points of ``include/cfgzip.h`` by way of the ctypes binding. A state
holds what such a program holds between two decode steps: a context with its partitions loaded, the class
masks of the grammar engine, the language model's logits and the result buffers it keeps. The logits are
masked in place, and masking them again gives the same results, so a pass can be repeated on one state.

Kinds of case
  greedy    cfgzip_masked_logsoftmax_argmax: the fused decode step (expand, mask, normalise, choose, map)
  mask      cfgzip_expand_mask, cfgzip_mask_logits, cfgzip_map_tokens: for a program with a sampler of its own
  sample    cfgzip_masked_sample and, with top-k or top-p, cfgzip_masked_sample_filtered
  multi     cfgzip_multi_mask_logsoftmax_argmax: one logits row under several grammar states
  host      cfgzip_decode_step_host: logits and masks in pinned host memory, results back on the host
  offline   grammar and vocabulary to a loaded partition (signatures on the host, grouping on the GPU)
"""
import numpy as np
import torch

from paper_2605_29986_b200 import binding as cz


# ---------------------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------------------
def listed():
    return [
        # one request, a small vocabulary: nothing but latency
        {"name": "greedy-f32-v32000-b1", "kind": "greedy", "V": 32000, "K": 256, "B": 1, "dtype": "f32",
         "density": 0.3, "grammars": 1},
        # the batch the decode-step metric is quoted on
        {"name": "greedy-bf16-v128256-b32", "kind": "greedy", "V": 128256, "K": 2048, "B": 32, "dtype": "bf16",
         "density": 0.1, "grammars": 1},
        # f32 logits, rows between almost nothing and almost everything allowed, all log-probabilities asked for
        # (beam search, log-probabilities reported to the client)
        {"name": "greedy-f32-v151936-b128-logp", "kind": "greedy", "V": 151936, "K": 4096, "B": 128, "dtype": "f32",
         "density": 0.0, "grammars": 1, "full": True},
        # a batch that serves eight grammars at once, large classes and many of them; the rows keep their grammars
        {"name": "greedy-bf16-v256000-b256-grammars", "kind": "greedy", "V": 256000, "K": 16384, "B": 256,
         "dtype": "bf16", "density": 0.0, "grammars": 8, "planned": True},
        # an odd vocabulary (tokens added to a tokenizer) with rows packed end to end
        {"name": "greedy-bf16-v100003-b48-odd", "kind": "greedy", "V": 100003, "K": 1500, "B": 48, "dtype": "bf16",
         "density": 0.2, "grammars": 1, "tight": True},
        # rows that allow a handful of classes only: structural characters, keywords
        {"name": "sparse-f32-v128256-b1024", "kind": "greedy", "V": 128256, "K": 512, "B": 1024, "dtype": "f32",
         "classes": 5, "grammars": 1},
        # mask only, for a program that samples by itself
        {"name": "mask-bf16-v128256-b512", "kind": "mask", "V": 128256, "K": 2048, "B": 512, "dtype": "bf16",
         "density": 0.1, "grammars": 1},
        # temperature 0.2, no filter
        {"name": "sample-bf16-v128256-b32", "kind": "sample", "V": 128256, "K": 2048, "B": 32, "dtype": "bf16",
         "density": 0.1, "grammars": 1, "temperature": 0.2, "top_k": 0, "top_p": 1.0},
        # the customary filters at a customary temperature
        {"name": "sample-bf16-v151936-b64-filtered", "kind": "sample", "V": 151936, "K": 4096, "B": 64, "dtype": "bf16",
         "density": 0.1, "grammars": 1, "temperature": 0.7, "top_k": 50, "top_p": 0.9},
        # speculative decoding: eight rows, sixteen candidate continuations each
        {"name": "multi-bf16-v128256-b8x16", "kind": "multi", "V": 128256, "K": 2048, "B": 8, "masks": 16,
         "dtype": "bf16", "density": 0.1, "grammars": 1},
        # everything on the host: copies in, step, results out
        {"name": "host-bf16-v128256-b32", "kind": "host", "V": 128256, "K": 2048, "B": 32, "dtype": "bf16",
         "density": 0.1, "grammars": 1},
        # once per tokenizer and grammar: signatures, grouping, loading
        {"name": "offline-v128256", "kind": "offline", "V": 128256},
    ]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw_one(rng)
        if _cost(case) <= most:
            return case


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _draw_one(rng):
    kind = rng.choice(("greedy", "greedy", "greedy", "mask", "sample", "sample", "multi", "host", "offline"))
    if kind == "offline":
        return {"kind": kind, "V": _log_uniform(rng, 8000, 128256)}
    V = _log_uniform(rng, 20000, 256000)
    tight = rng.random() < 0.25  # rows packed end to end; else the head is padded as language models pad theirs
    if not tight and rng.random() < 0.5:
        V = (V + 63) // 64 * 64
    case = {"kind": kind, "V": V, "K": min(_log_uniform(rng, 256, 16384), V // 8), "dtype": rng.choice(("bf16", "bf16", "f32")),
            "density": rng.choice((0.0, 0.01, 0.1, 0.3, 0.9)), "grammars": 1, "tight": tight}
    if kind == "greedy":
        case["B"] = _log_uniform(rng, 1, 1024)
        case["full"] = rng.random() < 0.2
        if rng.random() < 0.2:
            case["classes"] = rng.randint(1, 8)
        if case["B"] >= 4 and rng.random() < 0.25:
            case["grammars"] = rng.randint(2, 8)
            case["planned"] = rng.random() < 0.5
    elif kind == "mask":
        case["B"] = _log_uniform(rng, 1, 1024)
    elif kind == "sample":
        case["B"] = _log_uniform(rng, 8, 512)
        case["temperature"] = rng.choice((0.2, 0.7, 1.0))
        case["top_k"] = rng.choice((0, 0, 20, 50))
        case["top_p"] = rng.choice((1.0, 1.0, 0.9, 0.95))
    elif kind == "multi":
        case["tight"] = False  # the call takes 16-byte aligned rows only
        case["B"] = _log_uniform(rng, 1, 32)
        case["masks"] = _log_uniform(rng, 2, 32)
    else:
        case["tight"] = True  # host rows are dense: the call has no row stride
        case["B"] = _log_uniform(rng, 1, 64)
    return case


def _cost(case):
    """Bytes a pass moves, host bytes at the price of the bus."""
    return work(case)["bytes"] * (20 if case["kind"] == "host" else 1)


def _words(n):
    return (n + 31) // 32


def _elem(case):
    return 2 if case["dtype"] == "bf16" else 4


def _stride(case):
    """Elements from one logits row to the next: the vocabulary itself, or padded to a multiple of 64."""
    return case["V"] if case.get("tight") else (case["V"] + 63) // 64 * 64


def work(case):
    """What a pass cannot do without: every input read once, every output written once. A disallowed logit need not be
    read, which matters where hardly any is allowed; the token -> class vector counts as 16 bits per token."""
    V, kind = case["V"], case["kind"]
    if kind == "offline":
        # token bytes and offsets in; class of every token, representatives, class lists, signatures out and in again
        return {"bytes": float(V * (6 + 8 + 4 + 4 + 4 + 4 + 2 * 4 * _SIGNATURE_WORDS)), "flops": float(V * 8)}
    B, K, es = case["B"], case["K"], _elem(case)
    vm, cm, logits, classes = 4 * _words(V), 4 * _words(K), V * es, case["grammars"] * 2 * V
    if kind == "multi":
        M = case["masks"]
        return {"bytes": float(B * (logits + M * (vm + cm + 16)) + classes), "flops": float(3 * B * M * V)}
    if kind == "mask":
        return {"bytes": float(B * (2 * logits + 2 * vm + cm + 8) + classes), "flops": float(B * V)}
    if kind == "host":
        return {"bytes": float(B * (logits + vm + cm + 16) + classes), "flops": float(3 * B * V)}
    read = 1.0
    if "classes" in case:
        read = min(1.0, 0.5 * (1 + case["classes"]) / K)
        classes = 0
    full = 4 * V if case.get("full") else 0
    return {"bytes": float(B * ((1 + read) * logits + vm + cm + full + 20) + classes), "flops": float(3 * B * V)}


def tolerance(case):
    """Masks, masked logits, token ids and representatives are the same bits for every correct implementation. The
    normaliser is a 32-bit sum over up to 256000 terms; a log-probability z / T - lse is the difference of two numbers
    of the size of z / T, which is up to about 60 at temperature 0.2."""
    if case["kind"] == "offline":
        return "exact"
    return {"rel": 1e-4, "max": 1e-3} if case["kind"] == "sample" else {"rel": 1e-5, "max": 1e-4}


# ---------------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------------
class State:
    """A context and the buffers around it; the context goes with the object."""

    def __init__(self, case):
        self.case = case
        self.ctx = cz.cfgzip_create(torch.cuda.current_device())
        self.stream = torch.cuda.current_stream().cuda_stream

    def __del__(self):
        if getattr(self, "grammar", 0):
            cz.cfgzip_grammar_destroy(self.grammar)
        if getattr(self, "ctx", 0):
            cz.cfgzip_destroy(self.ctx)


def _partition(V, K, heavy, rs):
    """Class sizes by Zipf's law, members scattered over the vocabulary, lowest token id as representative. `heavy`: one
    class holds 60 % of the vocabulary (the tokens no rule of the grammar can use)."""
    first = int(0.6 * V) if heavy else 0
    n = K - 1 if heavy else K
    w = np.arange(1, n + 1) ** (-1.3 if heavy else -1.1)
    sizes = 1 + np.floor(w / w.sum() * (V - first - n)).astype(np.int64)
    sizes[: V - first - int(sizes.sum())] += 1
    sizes = rs.permutation(sizes)
    if heavy:
        sizes = np.concatenate([[first], sizes])
    c = np.empty(V, dtype=np.int32)
    c[rs.permutation(V)] = np.repeat(np.arange(K, dtype=np.int32), sizes)
    r = np.empty(K, dtype=np.int32)
    r[c[::-1]] = np.arange(V - 1, -1, -1, dtype=np.int32)  # the last write of a class is its lowest id
    return c, r


def _class_masks(case, rows, gen):
    """Packed class masks [rows, KW]: every class allowed with the case's density (0: a density of its own for every
    row), or 1 .. `classes` classes per row."""
    K, KW = case["K"], _words(case["K"])
    u = torch.rand((rows, K), generator=gen, device="cuda")
    if "classes" in case:
        n = torch.randint(1, case["classes"] + 1, (rows, 1), generator=gen, device="cuda")
        bits = u.argsort(dim=1).argsort(dim=1) < n
    else:
        p = case["density"] or torch.rand((rows, 1), generator=gen, device="cuda")
        bits = u < p
        bits[:, 0] |= ~bits.any(dim=1)  # the engine never leaves a row without a class
    padded = torch.zeros((rows, KW * 32), dtype=torch.int64, device="cuda")
    padded[:, :K] = bits
    words = (padded.view(rows, KW, 32) << torch.arange(32, device="cuda")).sum(dim=2)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32).contiguous()


def _logits(case, gen):
    """Normal logits, with fifty tokens per row the model is keen on."""
    B, V = case["B"], case["V"]
    z = torch.empty((B, _stride(case)), dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32, device="cuda")
    z.normal_(0.0, 2.0, generator=gen)
    keen = torch.randint(0, V, (B, 50), generator=gen, device="cuda")
    z.scatter_(1, keen, z.gather(1, keen) + 4.0)
    return z


def prepare(case, seed):
    if case["kind"] == "offline":
        return _prepare_offline(case, seed)
    s = State(case)
    rs = np.random.RandomState(seed % (1 << 32))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    V, K, B = case["V"], case["K"], case["B"]
    rows = B * case.get("masks", 1)
    s.code = cz.BF16 if case["dtype"] == "bf16" else cz.F32
    heavy = case["grammars"] > 1
    s.parts = []
    for _ in range(case["grammars"]):
        c, r = _partition(V, K, heavy, rs)
        s.parts.append(cz.cfgzip_load_partition(s.ctx, c, V, r, K, s.stream))
    s.row_part = None
    if heavy:
        s.row_part = torch.tensor(rs.randint(0, case["grammars"], B), dtype=torch.int32, device="cuda")
    s.masks = _class_masks(case, rows, gen)
    s.logits = _logits(case, gen)
    s.mode = cz.SPARSE if "classes" in case else cz.AUTO
    device = dict(device="cuda")
    if case["kind"] == "host":
        s.masks = s.masks.cpu().pin_memory()
        s.logits = s.logits.cpu().pin_memory()
        device = dict(pin_memory=True)
    s.vocab_mask = torch.zeros((rows, _words(V)), dtype=torch.int32, **device)
    s.token, s.rep = (torch.zeros(rows, dtype=torch.int32, **device) for _ in range(2))
    s.logp, s.lse = (torch.zeros(rows, dtype=torch.float32, **device) for _ in range(2))
    s.full = torch.zeros((B, V), dtype=torch.float32, device="cuda") if case.get("full") else None
    if case["kind"] == "sample":
        s.u = torch.rand(B, generator=gen, device="cuda")
        s.inv_temperature = 1.0 / case["temperature"]
    if case["kind"] == "mask":  # what the program's own sampler chose
        s.token = torch.randint(0, V, (B,), generator=gen, device="cuda", dtype=torch.int32)
    if case.get("planned"):
        cz.cfgzip_plan_rows(s.ctx, s.parts[0], s.row_part, B, s.stream)
        s.row_part_of_step = cz.ROWS_AS_PLANNED
    else:
        s.row_part_of_step = s.row_part
    return s


_SIGNATURE_WORDS = 64  # integers per signature row: the longest displacement of the vocabulary below has fewer


def _json_grammar():
    """JSON values without white space, character by character, in Greibach normal form: strings over the printable
    characters, integers, nested arrays and objects. (heads, terminals, offsets, symbols)"""
    names = ["V", "S", "N", "A", "T", "E", "M", "C", "W", "U", "P"]
    V, S, N, A, T, E, M, C, W, U, P = range(len(names))
    rules = []

    def value(head, tail):
        rules.append((head, '"', [S] + tail))
        for d in "0123456789":
            rules.append((head, d, tail))
            rules.append((head, d, [N] + tail))
        rules.append((head, "[", [A] + tail))
        rules.append((head, "{", [M] + tail))

    value(V, [])
    for code in range(32, 127):
        if chr(code) not in '"\\':
            rules.append((S, chr(code), [S]))
    rules.append((S, '"', []))
    for d in "0123456789":
        rules.append((N, d, []))
        rules.append((N, d, [N]))
    rules.append((A, "]", []))
    value(A, [T])
    rules.append((T, "]", []))
    rules.append((T, ",", [E]))
    value(E, [T])
    rules.append((M, "}", []))
    rules.append((M, '"', [S, C]))
    rules.append((C, ":", [W]))
    value(W, [U])
    rules.append((U, "}", []))
    rules.append((U, ",", [P]))
    rules.append((P, '"', [S, C]))
    heads = np.array([h for h, _, _ in rules], dtype=np.int32)
    terms = np.array([ord(t) for _, t, _ in rules], dtype=np.uint8)
    off = np.cumsum([0] + [len(b) for _, _, b in rules]).astype(np.int32)
    symbols = np.array([x for _, _, b in rules for x in b], dtype=np.int32)
    return len(names), heads, terms, off, symbols


def _vocabulary(V, rs):
    """Words with and without a leading space, numbers, runs of punctuation, bytes of other scripts: token bytes and
    offsets, about as long as the tokens of a byte-pair encoding."""
    letters = b"etaoinshrdlcumwfgypbvkjxqzETAOINSHRDLC"
    tables = [letters, letters, b"0123456789", b'":,{}[]":,{}[] _-.', bytes(range(192, 224))]
    kind = rs.choice(len(tables), V, p=[0.45, 0.3, 0.05, 0.08, 0.12])
    longest = np.array([12, 12, 3, 3, 6])[kind]
    length = 1 + (rs.random_sample(V) ** 1.5 * longest).astype(np.int64).clip(max=longest - 1)
    off = np.concatenate([[0], np.cumsum(length)]).astype(np.int64)
    table = np.zeros((len(tables), 64), dtype=np.uint8)
    size = np.zeros(len(tables), dtype=np.int64)
    for i, t in enumerate(tables):
        table[i, : len(t)] = np.frombuffer(t, dtype=np.uint8)
        size[i] = len(t)
    of_byte = np.repeat(kind, length)
    flat = table[of_byte, (rs.random_sample(len(of_byte)) * size[of_byte]).astype(np.int64)]
    flat[off[:-1][(kind == 1) & (length > 1)]] = ord(" ")
    return np.ascontiguousarray(flat), off, length.astype(np.int32)


def _prepare_offline(case, seed):
    s = State(case)
    V = case["V"]
    n, heads, terms, off, symbols = _json_grammar()
    s.grammar = cz.cfgzip_grammar_create(n, 0, heads, terms, off, symbols)
    s.bytes, s.off, length = _vocabulary(V, np.random.RandomState(seed % (1 << 32)))
    s.signatures = torch.zeros((V, _SIGNATURE_WORDS), dtype=torch.int32, pin_memory=True)
    s.length = torch.from_numpy(length).cuda()
    s.d_signatures = torch.zeros((V, _SIGNATURE_WORDS), dtype=torch.int32, device="cuda")
    s.c, s.r = (torch.zeros(V, dtype=torch.int32, device="cuda") for _ in range(2))
    s.n_classes = torch.zeros(1, dtype=torch.int32, device="cuda")
    s.class_off = torch.zeros(V + 1, dtype=torch.int32, device="cuda")
    s.class_tok = torch.zeros(V, dtype=torch.int32, device="cuda")
    return s


# ---------------------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------------------
def run(s):
    return _RUN[s.case["kind"]](s)


def _run_greedy(s):
    c = s.case
    cz.cfgzip_masked_logsoftmax_argmax(s.ctx, s.parts[0], s.row_part_of_step, s.masks, s.masks.shape[1], s.logits, s.code,
                                       s.logits.shape[1], c["B"], s.vocab_mask, s.vocab_mask.shape[1], s.token, s.rep,
                                       s.logp, s.lse, s.full, s.mode, s.stream)
    return [s.logits, s.vocab_mask, s.token, s.rep, s.logp, s.lse, s.full]


def _run_mask(s):
    c = s.case
    cz.cfgzip_expand_mask(s.ctx, s.parts[0], s.row_part_of_step, s.masks, s.masks.shape[1], s.vocab_mask,
                          s.vocab_mask.shape[1], c["B"], s.mode, s.stream)
    cz.cfgzip_mask_logits(s.ctx, s.logits, s.code, s.logits.shape[1], c["B"], c["V"], s.vocab_mask,
                          s.vocab_mask.shape[1], s.stream)
    cz.cfgzip_map_tokens(s.ctx, s.parts[0], s.row_part_of_step, s.token, s.rep, c["B"], s.stream)
    return [s.logits, s.vocab_mask, s.rep]


def _run_sample(s):
    c = s.case
    if c["top_k"] > 0 or c["top_p"] < 1.0:
        cz.cfgzip_masked_sample_filtered(s.ctx, s.parts[0], s.row_part_of_step, s.masks, s.masks.shape[1], s.logits,
                                         s.code, s.logits.shape[1], c["B"], s.vocab_mask, s.vocab_mask.shape[1], s.u,
                                         s.inv_temperature, c["top_k"], c["top_p"], s.token, s.rep, s.logp, s.lse,
                                         s.mode, s.stream)
    else:
        cz.cfgzip_masked_sample(s.ctx, s.parts[0], s.row_part_of_step, s.masks, s.masks.shape[1], s.logits, s.code,
                                s.logits.shape[1], c["B"], s.vocab_mask, s.vocab_mask.shape[1], s.u, s.inv_temperature,
                                s.token, s.rep, s.logp, s.lse, s.mode, s.stream)
    return [s.logits, s.vocab_mask, s.token, s.rep, s.logp, s.lse]


def _run_multi(s):
    c = s.case
    cz.cfgzip_multi_mask_logsoftmax_argmax(s.ctx, s.parts[0], s.masks, s.masks.shape[1], c["masks"], s.logits, s.code,
                                           s.logits.shape[1], c["B"], s.vocab_mask, s.vocab_mask.shape[1], s.token, s.rep,
                                           s.logp, s.lse, s.stream)
    return [s.vocab_mask, s.token, s.rep, s.logp, s.lse]


def _run_host(s):
    cz.cfgzip_decode_step_host(s.ctx, s.parts[0], None, s.masks, s.masks.shape[1], s.logits, s.code, s.case["B"], None,
                               s.vocab_mask, s.token, s.rep, s.logp, s.lse, s.mode, s.stream)
    return [s.vocab_mask, s.token, s.rep, s.logp, s.lse]


def _run_offline(s):
    V = s.case["V"]
    status = cz.cfgzip_displacement_signatures(s.grammar, s.bytes, s.off, V, _SIGNATURE_WORDS, s.signatures)
    if status != cz.OK:
        raise RuntimeError("a displacement does not fit its signature row")
    s.d_signatures.copy_(s.signatures, non_blocking=True)
    cz.cfgzip_group_tokens(s.d_signatures, _SIGNATURE_WORDS, s.length, V, s.c, s.r, s.n_classes, s.class_off, s.class_tok,
                           s.stream)
    K = int(s.n_classes.item())
    part = cz.cfgzip_load_partition(s.ctx, s.c.cpu(), V, s.r[:K].cpu(), K, s.stream)
    cz.cfgzip_free_partition(s.ctx, part)  # the next pass stands for the next grammar
    return [s.signatures, s.c, s.r, s.n_classes, s.class_off, s.class_tok]


_RUN = {"greedy": _run_greedy, "mask": _run_mask, "sample": _run_sample, "multi": _run_multi, "host": _run_host,
        "offline": _run_offline}
