"""What a user of this framework has it do, as measurable cases: paged MLA decode calls through the binding.

Every case is one decode call on device tensors that a serving loop keeps (query rows, paged latent cache, block
table, lengths, output buffers, workspace).  A case is described by

  entry      "workspace" (mla_decode), "static" (mla_decode_static) or "fp8" (mla_decode_fp8, E4M3 cache)
  B, Sq, H   sequences, query tokens per sequence (more than one: speculative tokens), query heads
  n_lo, n_hi range of the sequences' lengths in keys (equal: all sequences have that length)
  n_seed     picks the lengths inside the range
  rising     the keys carry a logit offset that rises in steps from -30 to +30 along the sequence, so that the
             running maximum keeps moving (otherwise the logits are those of N(0, 1) queries and keys)

Pages (64 keys) lie in the cache in random order, as after some time of serving.
"""
import math
import random

import torch

from paper_2509_25224_b200 import binding

PAGE, D_QK, D_V = 64, 576, 512
SCALE = 1.0 / math.sqrt(192.0)
KV_SCALE = 1.0 / 64.0                # dequantisation factor of the E4M3 caches: N(0, 1) values land around +-64 of +-448
MAX_KEYS = 96 * 16384                # keys of the largest case's cache


def case(name, B, Sq, H, n_lo, n_hi=None, n_seed=0, entry="workspace", rising=False):
    c = {"entry": entry, "B": B, "Sq": Sq, "H": H, "n_lo": n_lo, "n_hi": n_lo if n_hi is None else n_hi, "n_seed": n_seed, "rising": rising}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the smallest call: one short sequence, 16 heads; launches and host work are all there is
        case("tiny", 1, 1, 16, 256),
        # one user's stream in a loop that must not enter the allocator; a length that is no multiple of anything
        case("one-stream", 1, 1, 128, 2531, entry="static"),
        # the start of many chats: more sequences than the GPU has room for clusters, each a few pages
        case("short-batch", 192, 1, 128, 1, 512, 11),
        # the plain decode step of a medium batch at a medium length
        case("batch32-4k", 32, 1, 128, 4096),
        # the same work sharded over eight GPUs by heads: 16 heads are left here, every GPU reads the whole cache
        case("heads16-ragged", 32, 1, 16, 1024, 8192, 12),
        # logits whose maximum keeps rising: every tile moves the reference of the online softmax
        case("rising-16k", 16, 1, 128, 16384, rising=True),
        # a large batch of short contexts, one query token
        case("batch96-2k", 96, 1, 128, 2048),
        # speculative decoding: two query tokens per sequence, ragged lengths
        case("spec2-ragged", 64, 2, 128, 1024, 8192, 13),
        # a few very long contexts: every sequence is split over many clusters and merged
        case("spec2-64k", 4, 2, 128, 65536),
        # the largest: throughput serving, full batch, long contexts, two query tokens
        case("spec2-batch96-16k", 96, 2, 128, 16384),
        # E4M3 cache, one query token, medium batch
        case("fp8-batch32-4k", 32, 1, 128, 4096, entry="fp8"),
        # E4M3 cache, two query tokens, ragged lengths
        case("fp8-spec2-ragged", 32, 2, 128, 512, 8192, 14, entry="fp8"),
    ]


def log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choices(["workspace", "static", "fp8"], [6, 1, 2])[0]
    Sq = rng.choices([1, 2, rng.randint(3, 8)], [5, 3, 1])[0]
    H = rng.choices([128, 64, 32, 16, rng.randint(8, 128)], [6, 1, 1, 1, 1])[0]
    n_hi = log_uniform(rng, 32, 65536)
    n_lo = n_hi if rng.random() < 0.4 else rng.randint(1, n_hi)
    # one block of 128 query rows over all keys is the unit of cost; a quarter of it on the E4M3 cache, whose calls take longer
    most_keys = MAX_KEYS / max(1.0, math.ceil(Sq * H / 128) / 2.0)
    if entry == "fp8":
        most_keys /= 4.0
    B = log_uniform(rng, 1, max(1.0, min(200.0, most_keys / n_hi)))
    return case(None, B, Sq, H, n_lo, n_hi, rng.randrange(1 << 20), entry, entry != "fp8" and rng.random() < 0.15)


def lengths(case):
    r = random.Random(case["n_seed"])
    return [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["B"])]


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    B, Sq, H, lens = case["B"], case["Sq"], case["H"], lengths(case)
    pages = [(n + PAGE - 1) // PAGE for n in lens]
    total, width = sum(pages), max(pages)

    def normal(shape, dtype, gain=1.0):
        out = torch.empty(shape, dtype=dtype, device=dev)
        for part in out.view(-1).split(1 << 27):
            part.copy_(torch.randn(part.shape, generator=gen, device=dev).mul_(gain).clamp_(-448.0, 448.0))
        return out

    q = normal((B, Sq, H, D_QK), torch.bfloat16)
    fp8 = case["entry"] == "fp8"
    kv = normal((total, PAGE, D_QK), torch.float8_e4m3fn, 1.0 / KV_SCALE).view(torch.uint8) if fp8 else normal((total, PAGE, D_QK), torch.bfloat16)
    # the sequences' pages, in order, are the entries of a permutation of the cache's pages
    place = torch.randperm(total, generator=gen, device=dev).to(torch.int32)
    count = torch.tensor(pages, device=dev)
    owner = torch.repeat_interleave(torch.arange(B, device=dev), count, output_size=total)
    index = torch.arange(total, device=dev) - (count.cumsum(0) - count)[owner]
    table = torch.full((B, width), -1, dtype=torch.int32, device=dev)
    table[owner, index] = place
    seqlens = torch.tensor(lens, dtype=torch.int32, device=dev)
    if case["rising"]:
        gain = 4.0
        key = index[:, None] * PAGE + torch.arange(PAGE, device=dev)
        step = (32 * key // seqlens[owner][:, None].long()).clamp_(max=31)
        q[..., D_V] = gain
        kv[place.long(), :, D_V] = ((-30.0 + 60.0 / 31.0 * step) / (gain * SCALE)).to(torch.bfloat16)
    size = binding.fp8_workspace_size if fp8 else binding.workspace_size
    return {
        "entry": case["entry"], "q": q, "kv": kv, "table": table, "seqlens": seqlens,
        "out": torch.empty((B, Sq, H, D_V), dtype=torch.bfloat16, device=dev),
        "lse": torch.empty((B, Sq, H), dtype=torch.float32, device=dev),
        "workspace": None if case["entry"] == "static" else torch.empty(size(B, Sq, H, width, dev.index), dtype=torch.uint8, device=dev),
    }


def run(state):
    s = state
    if s["entry"] == "fp8":
        return binding.mla_decode_fp8(s["q"], s["kv"], KV_SCALE, s["table"], s["seqlens"], SCALE, s["out"], s["lse"], s["workspace"])
    if s["entry"] == "static":
        binding.mla_decode_static(s["q"], s["kv"], s["table"], s["seqlens"], SCALE, s["out"], s["lse"])
        return s["out"], s["lse"]
    return binding.mla_decode(s["q"], s["kv"], s["table"], s["seqlens"], SCALE, s["out"], s["lse"], s["workspace"])


def work(case):
    lens = lengths(case)
    rows = case["B"] * case["Sq"] * case["H"]
    key_bytes = D_QK * (1 if case["entry"] == "fp8" else 2)
    table_bytes = 4 * (sum((n + PAGE - 1) // PAGE for n in lens) + len(lens))
    return {"bytes": sum(lens) * key_bytes + rows * (2 * D_QK + 2 * D_V + 4) + table_bytes,
            "flops": 2.0 * case["Sq"] * case["H"] * sum(lens) * (D_QK + D_V)}


def tolerance(case):
    return {"rel": 8e-3, "max": 8e-2}
