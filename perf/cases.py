"""What this library is measured on: the calls its users make, over the sizes they make them at.

Every case is one use of the public Python binding (``paper_2607_29678_b200``) on seeded synthetic text of the shapes in
``workloads``.  ``op`` names the use:

  request   ``Vocab.encode``: one request's text on the device -> token ids on the device (a prompt on its way to the model)
  batch     ``Vocab.encode_batch``: independent documents, concatenated, in one call
  host      ``Vocab.encode_host_into``: host text -> host ids, on pinned buffers or on ordinary (pageable) ones
  chat      ``Vocab.encode_added``: a transcript whose role markers are added tokens
  spans     ``Vocab.encode`` and ``Vocab.spans``: ids with the byte and character offset of every token
  session   ``Session``: a conversation from its creation (a context, then its turns, appended one by one) to the reading of
            its records and its end

``pattern`` is the pre-tokenization pattern (0 cl100k-style, 1 o200k-style, 2 single digits, 3 three splitters), ``merges``
the size of the stored vocabulary, ``kind`` the generator's kind of text (0 prose / code / JSON, 1 the same with accented,
Cyrillic and CJK text, emoji and CRLF, 2 agent transcript, 3 transcript with CJK and very long runs, 4 combining marks,
5 Thai-like text without blanks).
"""
import functools
import math

import numpy as np
import torch

import paper_2607_29678_b200 as tt
import workloads as wl

MARKERS = ["<|system|>", "<|user|>", "<|assistant|>", "<|tool|>", "<|endoftext|>"]
MARKER_ID0 = 300_000

# bytes per character of each kind of text, and tokens per byte (with the larger vocabularies), for work()
BYTES_PER_CHAR = (1.0, 1.07, 1.0, 1.35, 1.28, 2.89)
TOKENS_PER_BYTE = (0.19, 0.22, 0.19, 0.24, 0.91, 0.99)
# most bytes per character of each kind: buffers are sized once, for the longest text of their case
MOST_BYTES_PER_CHAR = (1, 2, 1, 4, 2, 4)


def listed():
    return [
        # A short chat message: the smallest request of the benchmark, where launches and latency are everything.
        {"name": "request 4K chars", "op": "request", "kind": 0, "chars": 4_000, "pattern": 0, "merges": 4_096},
        # A document or a long prompt with non-ASCII text and CRLF lines.
        {"name": "request 100K unicode", "op": "request", "kind": 1, "chars": 100_000, "pattern": 0, "merges": 32_000},
        # The headline request: a million characters of agent transcript.
        {"name": "request 1M transcript", "op": "request", "kind": 2, "chars": 1_000_000, "pattern": 0, "merges": 100_000},
        # The largest single request: CJK text, 64 KB blank runs, 20,000-digit numbers, 50 KB punctuation runs.
        {"name": "request 3M long runs", "op": "request", "kind": 3, "chars": 3_000_000, "pattern": 1, "merges": 199_744},
        # A script without blanks that the vocabulary knows little of: nearly a token per byte.
        {"name": "request 1M thai-like", "op": "request", "kind": 5, "chars": 1_000_000, "pattern": 1, "merges": 199_744},
        # Bulk ingestion: 256 requests of 10,000 to 3,000,000 characters (132 MB) in one call.
        {"name": "batch 256 requests", "op": "batch", "kind": 2, "docs": 256, "chars": 350_000, "pattern": 0, "merges": 100_000},
        # A serving step's worth of short messages in one call.
        {"name": "batch 1000 messages", "op": "batch", "kind": 1, "docs": 1_000, "chars": 900, "pattern": 1, "merges": 199_744},
        # A server whose texts arrive in pinned host memory and whose ids leave through it.
        {"name": "host 1M pinned", "op": "host", "kind": 2, "chars": 1_000_000, "pattern": 0, "merges": 100_000, "pinned": True},
        # A script that hands over an ordinary array and wants an array back.
        {"name": "host 100K pageable", "op": "host", "kind": 1, "chars": 100_000, "pattern": 3, "merges": 32_000, "pinned": False},
        # A conversation with its role markers as special tokens, under the whole-piece (ignore_merges) rule.
        {"name": "chat 300K markers", "op": "chat", "kind": 2, "chars": 300_000, "pattern": 0, "merges": 100_000, "ignore_merges": True},
        # Ids with offsets, as a training or annotation pipeline wants them.
        {"name": "spans 1M", "op": "spans", "kind": 2, "chars": 1_000_000, "pattern": 2, "merges": 100_000},
        # A conversation of 16 turns on top of a 60,000-character context.
        {"name": "session 16 turns", "op": "session", "kind": 2, "chars": 60_000, "turns": 16, "turn_chars": 1_500, "pattern": 0, "merges": 100_000},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text_options(rng, kinds):
    kind = rng.choice(kinds)
    pattern = 1 if kind >= 3 else rng.choice((0, 0, 1, 2, 3))            # the kinds of the o200k-style configurations
    merges = 199_744 if pattern == 1 else rng.choice((4_096, 32_000, 100_000))
    return {"kind": kind, "pattern": pattern, "merges": merges}


def draw(rng):
    op = rng.choice(("request", "request", "request", "batch", "batch", "host", "chat", "spans", "session"))
    if op == "request":
        c = _text_options(rng, (0, 1, 2, 2, 3, 4, 5))
        c["chars"] = _log_uniform(rng, 1_000, 1_000_000 if c["kind"] >= 4 else 3_000_000)
    elif op == "batch":
        c = _text_options(rng, (0, 1, 2, 2))
        c["docs"] = _log_uniform(rng, 16, 1_000)
        c["chars"] = _log_uniform(rng, 300, min(350_000, 60_000_000 // c["docs"]))
    elif op == "host":
        c = _text_options(rng, (0, 1, 2))
        c["chars"] = _log_uniform(rng, 4_000, 1_000_000)
        c["pinned"] = rng.random() < 0.5
    elif op == "chat":
        c = _text_options(rng, (2,))
        c["chars"] = _log_uniform(rng, 4_000, 1_000_000)
        c["ignore_merges"] = rng.random() < 0.5
    elif op == "spans":
        c = _text_options(rng, (0, 1, 2))
        c["chars"] = _log_uniform(rng, 4_000, 1_000_000)
    else:
        c = _text_options(rng, (0, 1, 2))
        c["chars"] = _log_uniform(rng, 4_000, 200_000)
        c["turns"] = rng.randint(2, 12)
        c["turn_chars"] = _log_uniform(rng, 200, 4_000)
    return dict(c, op=op)


@functools.lru_cache(maxsize=None)
def _vocab(merges, pattern, ignore_merges, markers):
    """A user's program loads its vocabulary once and keeps it."""
    config = next(c for c in wl.CONFIGS.values() if c.n_merges == merges)
    table, byte_map = wl.load_vocab(config)
    v = tt.Vocab(table, byte_map, pattern, ignore_merges=ignore_merges)
    if markers:
        v.add_literals(MARKERS, [MARKER_ID0 + i for i in range(len(MARKERS))])
    return v


def _doc_lengths(case):
    # lognormal around the median, clipped as in the 256-request configuration; the same lengths for every seed
    m = case["chars"]
    return wl.batch_lengths(wl.BASE_SEED, case["docs"], m, 1.0, max(1.0, m / 35.0), m * 8.6)


def _buffers(v, n_bytes, n_docs=1):
    bufs = v.alloc(n_bytes, max_docs=n_docs)
    bufs["ids"].zero_()                                                    # the entries behind the count stay zero
    return bufs


def prepare(case, seed):
    op, kind, chars = case["op"], case["kind"], case["chars"]
    v = _vocab(case["merges"], case["pattern"], case.get("ignore_merges", False), op == "chat")
    base = 1_000_003 * (seed + 1)                                          # texts of one seed are no other seed's
    s = {"op": op, "vocab": v}
    if op == "batch":
        lengths = np.random.default_rng(seed).permutation(_doc_lengths(case))
        docs = [wl.generate(kind, base + i + 1, int(n)) for i, n in enumerate(lengths)]
        off = np.zeros(len(docs) + 1, dtype=np.int64)
        off[1:] = np.cumsum([d.size for d in docs])
        s["text"] = torch.from_numpy(np.concatenate(docs)).cuda()
        s["doc_off"] = torch.from_numpy(off).cuda()
        s["bufs"] = _buffers(v, int(lengths.sum()) * MOST_BYTES_PER_CHAR[kind], len(docs))
        return s
    most = chars * MOST_BYTES_PER_CHAR[kind]
    if op == "session":
        s["parts"] = [wl.generate(kind, base, chars)] + [wl.generate(kind, base + 1 + i, case["turn_chars"]) for i in range(case["turns"])]
        s["max_bytes"] = most + case["turns"] * case["turn_chars"] * MOST_BYTES_PER_CHAR[kind]
        s["ids"] = torch.zeros(s["max_bytes"], dtype=torch.int32, device="cuda")
        s["off"] = torch.zeros(s["max_bytes"] + 1, dtype=torch.int32, device="cuda")
        return s
    text = torch.from_numpy(wl.generate(kind, base, chars))
    if op == "host":
        ids = torch.zeros(most, dtype=torch.int32)
        s["text"], s["ids"] = (text.pin_memory(), ids.pin_memory()) if case["pinned"] else (text, ids)
        return s
    s["text"] = text.cuda()
    s["bufs"] = _buffers(v, most)
    if op == "spans":
        s["byte_off"] = torch.zeros(most + 1, dtype=torch.int32, device="cuda")
        s["char_off"] = torch.zeros(most + 1, dtype=torch.int32, device="cuda")
        s["span_status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        s["span_ws"] = torch.empty(int(tt.lib().tt_spans_workspace_bytes(v._h, most)), dtype=torch.uint8, device="cuda")
    return s


def run(state):
    v, op = state["vocab"], state["op"]
    if op == "host":
        n = v.encode_host_into(state["text"], state["ids"])
        return {"ids": state["ids"], "count": n}
    if op == "session":
        session = tt.Session(v, state["max_bytes"])
        for part in state["parts"]:
            session.append(part)
        ids, off, _ = session.records()
        session.close()
        state["ids"][:ids.numel()] = ids                                   # into the buffers that the model reads
        state["off"][:off.numel()] = off
        return {"ids": state["ids"], "byte_off": state["off"], "count": ids.numel()}
    text, bufs = state["text"], state["bufs"]
    if op == "batch":
        v.encode_batch(text, state["doc_off"], bufs)
        return {"ids": bufs["ids"], "ids_off": bufs["ids_off"], "status": bufs["status"]}
    if op == "chat":
        v.encode_added(text, bufs)
    else:
        v.encode(text, bufs)
    out = {"ids": bufs["ids"], "count": bufs["count"], "status": bufs["status"]}
    if op == "spans":
        v.spans(bufs["ids"], bufs["count"], text.numel(), state["byte_off"], state["char_off"], state["span_status"], workspace=state["span_ws"])
        out.update(byte_off=state["byte_off"], char_off=state["char_off"], span_status=state["span_status"])
    return out


def work(case):
    """The text once in, the ids (and offsets) once out."""
    op, kind = case["op"], case["kind"]
    chars = case["chars"]
    if op == "batch":
        chars = float(np.sum(_doc_lengths(case)))
    elif op == "session":
        chars += case["turns"] * case["turn_chars"]
    text = chars * BYTES_PER_CHAR[kind]
    tokens = text * TOKENS_PER_BYTE[kind]
    per_token = 12 if op == "spans" else 8 if op == "session" else 4
    return {"bytes": text + per_token * tokens + (16 * case["docs"] if op == "batch" else 0), "flops": 0}


def tolerance(case):
    """Token ids, counts and offsets are whole numbers with one right answer."""
    return "exact"
