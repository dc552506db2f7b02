"""Performance cases of the committed optimizer step: what a training job asks of
this library, through the Python entry points, over the range of sizes, table
shapes and options that it is used with.

A case is a dict:
  op       "commit" (AdamW step + digests), "verify" (read-only state digest),
           "step" (a commit and its verification, as after a recovery),
           "guard" (nonzero gradient words) or "upload" (a gradient bucket from
           page-locked host memory into the device's gradient buffers)
  layout   "f32" (fp32 master and moments, bf16 gradient and working copy) or
           "bf16" (parameters and moments kept in bf16)
  n        elements in all
  tensors  entries of the chunk table
  spread   natural logarithm of the largest entry's size over the smallest's
  unit     every entry's size is a multiple of this (128 for a model's matrices
           and norms, 1 for a table cut at odd places)
  packed   the state (for "upload": the host bucket) lies back to back in its
           allocation, as FSDP's flat shard does, while gradients and working
           copies start at 256-byte boundaries of theirs; otherwise all do
  goff     index of the first element in the flat model
  zero     the commit also zeroes the gradients
  step     the optimizer step
"""
import math
import random

import torch

import paper_2609_18178_gb300 as apc

ALIGN = 128  # elements: 256 bytes of bf16, 512 of fp32
LR, B1, B2, EPS, WD = 3e-4, 0.9, 0.95, 1e-8, 0.1  # apc.DEFAULT_HPARAMS
M32 = (1 << 32) - 1


def _case(op, n, tensors=1, layout="f32", spread=0.0, unit=1, packed=False, goff=0, zero=False, step=18, name=None):
    c = dict(op=op, layout=layout, n=n, tensors=tensors, spread=spread, unit=unit, packed=packed, goff=goff, zero=zero,
             step=step)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest calls: one short ragged shard across index 2^32 (the
        # smoke workload), where launches and latency are all there is.
        _case("commit", 100_003, goff=(1 << 32) - 50_000, step=3, name="commit_short_shard"),
        # A small model's flat shard, committed and verified: 29 MB of state.
        _case("step", 1 << 20, name="step_1m_shard"),
        # An ordinary model as a table of matrices and norms (152 M elements in
        # 146 tensors).
        _case("commit", 152_000_000, 146, spread=8.6, unit=128, step=10, name="commit_152m_table"),
        # One rank of 16 of a 7.25 B-parameter model, across index 2^32, with
        # the gradients zeroed at the committed boundary.
        _case("commit", 453_001_472, 21, spread=3.0, unit=128, goff=4_077_013_248, zero=True, step=5,
              name="commit_zero_rank_shard"),
        # A table of many small tensors (norms, biases, adapters), more than
        # one launch holds.
        _case("commit", 4_500_000, 1100, spread=5.0, name="commit_many_small"),
        # An odd-sized table whose state is one packed flat shard, while each
        # gradient and working copy has an allocation boundary of its own: the
        # buffers of most entries are not mutually 16-byte aligned.
        _case("commit", 60_000_000, 291, spread=6.0, packed=True, name="commit_packed_odd"),
        # The paper's own precision: a rank of 4, everything in bf16.
        _case("commit", 1_812_005_888, 74, layout="bf16", spread=3.0, unit=128, goff=1_812_005_888, step=5,
              name="commit_bf16_rank_shard"),
        # Verification after a recovery: fp32 state, many small tensors, bf16 state.
        _case("verify", 453_001_472, 21, spread=3.0, unit=128, goff=4_077_013_248, name="verify_rank_shard"),
        _case("verify", 4_500_000, 1100, spread=5.0, name="verify_many_small"),
        _case("verify", 1_812_005_888, 74, layout="bf16", spread=3.0, unit=128, goff=1_812_005_888,
              name="verify_bf16_rank_shard"),
        # The quiescence guard over a model's gradients.
        _case("guard", 152_000_000, 146, spread=8.6, unit=128, name="guard_152m_table"),
        # One packed gradient bucket of odd-sized tensors, host to device.
        _case("upload", 20_000_000, 146, spread=6.0, packed=True, name="upload_packed_bucket"),
    ]


def draw(rng):
    op = rng.choice(["commit", "commit", "commit", "verify", "verify", "step", "guard", "upload"])
    packed = rng.random() < 0.25 if op != "upload" else rng.random() < 0.5
    top = {"upload": 20_000_000, "guard": 450_000_000}.get(op, 60_000_000 if packed else 450_000_000)
    n = int(math.exp(rng.uniform(math.log(20_000), math.log(top))))
    tensors = max(1, min(int(math.exp(rng.uniform(0.0, math.log(1200)))), n // 256))
    spread = rng.uniform(0.5, 6.0)
    unit = 1 if packed else rng.choice([1, 8, 128])
    layout = rng.choice(["f32", "f32", "bf16"])
    return _case(op, n, tensors, layout, spread, unit, packed, goff=rng.randrange(1 << 33), zero=rng.random() < 0.3,
                 step=rng.randrange(1, 2000))


def _sizes(case):
    """The table's entry sizes: a function of the case alone."""
    t, n, unit = case["tensors"], case["n"], case["unit"]
    r = random.Random("%d/%d/%g" % (n, t, case["spread"]))
    w = [math.exp(case["spread"] * r.random()) for _ in range(t)]
    total = sum(w)
    sizes = [max(unit, int(n * x / total) // unit * unit) for x in w]
    big = max(range(t), key=sizes.__getitem__)
    sizes[big] = max(1, n - (sum(sizes) - sizes[big]))
    return sizes


def _places(sizes, packed):
    """Each entry's first element in its allocation, and the allocation's length."""
    at, off = [], 0
    for s in sizes:
        at.append(off)
        off += s if packed else -(-s // ALIGN) * ALIGN
    return at, off


def _layout(case):
    sizes = _sizes(case)
    at_s, len_s = _places(sizes, case["packed"])
    at_g, len_g = _places(sizes, False)
    goffs, g = [], case["goff"]
    for s in sizes:
        goffs.append(g)
        g += s
    return sizes, at_s, len_s, at_g, len_g, goffs


def _normal(n, sigma, gen, dtype):
    out = torch.empty(n, dtype=dtype, device="cuda")
    for a in range(0, n, 1 << 27):
        b = min(n, a + (1 << 27))
        out[a:b] = torch.randn(b - a, generator=gen, device="cuda").mul_(sigma)
    return out


def _inputs(case, seed):
    """The buffers of the case, with a training job's magnitudes: p of an
    initialised model, small moments, v a square, a gradient with exact zeros."""
    sizes, at_s, len_s, at_g, len_g, goffs = _layout(case)
    gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 17)
    sd = torch.float32 if case["layout"] == "f32" else torch.bfloat16
    op = case["op"]
    b = {}
    if op in ("commit", "verify", "step"):
        b["p"] = _normal(len_s, 0.02, gen, sd)
        b["m"] = _normal(len_s, 1e-4, gen, sd)
        b["v"] = _normal(len_s, 1e-3, gen, sd).square_()
        if case["layout"] == "f32":
            b["w"] = _normal(len_g, 0.02, gen, torch.bfloat16)
    if op != "verify":
        g = _normal(len_g, 1e-3, gen, torch.bfloat16)
        for a in range(0, len_g, 1 << 27):  # one in a hundred is an exact zero
            x = g[a:a + (1 << 27)]
            x.masked_fill_(torch.rand(x.numel(), generator=gen, device="cuda") < 0.01, 0.0)
        b["g"] = g
    return b


def prepare(case, seed):
    sizes, at_s, len_s, at_g, len_g, goffs = _layout(case)
    b = _inputs(case, seed)
    s = {"case": case, "b": b}
    view = lambda k, i: b[k][(at_s if k in "pmv" else at_g)[i]:][:sizes[i]]
    op, f32 = case["op"], case["layout"] == "f32"
    r = range(len(sizes))
    if op in ("commit", "step"):
        if f32:
            t = [apc.TensorEntry(view("p", i), view("m", i), view("v", i), view("g", i), view("w", i), goffs[i]) for i in r]
        else:
            t = [apc.TensorEntryBF16(view("p", i), view("m", i), view("v", i), view("g", i), goffs[i]) for i in r]
        s["table"] = apc.prepare_table(t)
        s["commit_out"] = torch.empty(4 if f32 else 3, dtype=torch.int64, device="cuda")
    if op in ("verify", "step"):
        if f32:
            e = [x for i in r for x in apc.state_buffers(view("p", i), view("m", i), view("v", i), view("w", i), goffs[i])]
        else:
            e = [x for i in r for x in apc.state_buffers_bf16(view("p", i), view("m", i), view("v", i), goffs[i])]
        s["buffers"] = apc.prepare_buffers(e)
        s["verify_out"] = torch.empty(4 if f32 else 3, dtype=torch.int64, device="cuda")
    if op == "guard":
        s["buffers"] = apc.prepare_buffers([apc.BufferEntry(view("g", i), 0, goffs[i], apc.BF16) for i in r])
        s["guard_out"] = torch.empty(1, dtype=torch.int64, device="cuda")
    if op == "upload":
        host = torch.empty(len_s, dtype=torch.bfloat16, pin_memory=True)
        whole = torch.empty(len_s, dtype=torch.bfloat16, device="cuda")
        for i in r:
            whole[at_s[i]:at_s[i] + sizes[i]] = view("g", i)
        host.copy_(whole)
        b["host"] = host
        b["g"].zero_()
        s["segments"] = apc.prepare_segments([apc.Segment(view("g", i), host[at_s[i]:at_s[i] + sizes[i]]) for i in r])
    return s


def run(state):
    """One pass.  The state is updated in place, so a repeated pass is the next
    step on the same gradient."""
    case, b, op = state["case"], state["b"], state["case"]["op"]
    f32 = case["layout"] == "f32"
    out = {}
    if op in ("commit", "step"):
        commit = apc.commit_step if f32 else apc.commit_step_bf16
        out["commit_digests"] = commit(state["table"], case["step"], out=state["commit_out"], zero_grad=case["zero"])
        out.update((k, b[k]) for k in ("p", "m", "v"))
        if f32:
            out["w"] = b["w"]
        if case["zero"]:
            out["g"] = b["g"]
    if op in ("verify", "step"):
        out["digests"] = apc.digest(state["buffers"], 4 if f32 else 3, out=state["verify_out"])
    if op == "guard":
        out["nonzero"] = apc.count_nonzero(state["buffers"], 1, out=state["guard_out"])
    if op == "upload":
        apc.upload(state["segments"])
        out["g"] = b["g"]
    return out


def work(case):
    """Bytes: p, m, v read and written, g read, w written (and g written when
    zeroed); the verified state or the guarded gradients read; the uploaded
    bytes read on the host side and written on the device's.  Operations: the
    update's 15 per element."""
    n, f32 = case["n"], case["layout"] == "f32"
    nbytes = flops = 0
    if case["op"] in ("commit", "step"):
        nbytes += n * ((28 if f32 else 14) + (2 if case["zero"] else 0))
        flops += 15 * n
    if case["op"] in ("verify", "step"):
        nbytes += n * (14 if f32 else 6)
    if case["op"] == "guard":
        nbytes += 2 * n
    if case["op"] == "upload":
        nbytes += 4 * n
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """The library's contract is identical bits: every operation of the update
    is one IEEE rounding in a fixed order, digests and counts are whole numbers
    and an upload moves bytes."""
    return "exact"


def _splitmix_sum(bits, goff, total):
    """total + the digest of one buffer's words (int64 tensor of zero-extended
    bits), mod 2^64, in wrapping int64 arithmetic."""
    i64 = lambda x: x - (1 << 64) if x >= (1 << 63) else x
    shr = lambda z, k: (z >> k) & ((1 << (64 - k)) - 1)
    g = (torch.arange(bits.numel(), device=bits.device, dtype=torch.int64) + goff) & M32
    z = (g << 32) + bits + i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
    z = z ^ shr(z, 31)
    return total + z.sum()


def _digest(buf, at, sizes, goffs):
    total = torch.zeros((), dtype=torch.int64, device="cuda")
    for a, n, g in zip(at, sizes, goffs):
        for c in range(0, n, 1 << 25):
            x = buf[a + c:a + min(n, c + (1 << 25))]
            bits = (x.view(torch.int32).to(torch.int64) & M32 if x.element_size() == 4
                    else x.view(torch.int16).to(torch.int64) & 0xFFFF)
            total = _splitmix_sum(bits, g + c, total)
    return total


def exact(case, seed):
    """The textbook decoupled AdamW in binary64 (the working copy as the
    unrounded parameter); digests of given words, counts and copied bytes as
    whole numbers.  Digests of computed words have no such value."""
    sizes, at_s, len_s, at_g, len_g, goffs = _layout(case)
    b = _inputs(case, seed)
    op, f32, t = case["op"], case["layout"] == "f32", case["step"]
    if op == "guard":
        return {"nonzero": torch.stack([sum((b["g"][a:a + n].view(torch.int16) != 0).sum() for a, n in zip(at_g, sizes))])}
    if op == "upload":
        out = torch.zeros_like(b["g"])
        for a, n in zip(at_g, sizes):
            out[a:a + n] = b["g"][a:a + n]
        return {"g": out.double()}
    if op == "verify":
        return {"digests": torch.stack([_digest(b[k], at_g if k == "w" else at_s, sizes, goffs)
                                        for k in ("pmvw" if f32 else "pmv")])}
    # gaps between aligned entries keep their contents
    out = {k: b[k].double() for k in ("pmvw" if f32 else "pmv")}
    for a, c, n in zip(at_s, at_g, sizes):
        for x in range(0, n, 1 << 27):
            s = slice(a + x, a + min(n, x + (1 << 27)))
            h = slice(c + x, c + min(n, x + (1 << 27)))
            p, m, v, g = out["p"][s], out["m"][s], out["v"][s], b["g"][h].double()
            m.mul_(B1).add_(g, alpha=1.0 - B1)
            v.mul_(B2).add_(g.square_(), alpha=1.0 - B2)
            den = (v / (1.0 - B2 ** t)).sqrt_().add_(EPS)
            u = (m / (1.0 - B1 ** t)).div_(den)
            p.mul_(1.0 - LR * WD).sub_(u, alpha=LR)
            if f32:
                out["w"][h] = p
    out["commit_digests"] = None
    if case["zero"]:
        g = b["g"].double()
        for c, n in zip(at_g, sizes):
            g[c:c + n] = 0
        out["g"] = g
    if op == "step":
        out["digests"] = None
    return out
