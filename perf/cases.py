"""The calls that a training run makes through this library, as cases that can be timed and compared.

A case is one model layout (transformer blocks, widths, vocabulary), a way its tensors lie in memory and
one path through the public entry points:

  decide   measure + select: the per-step question whether a layer has to be persisted.  Nothing has drifted far
           enough, which is what most steps of a run see.
  sums     the measure of a program that may not allocate (lc_measure_noalloc): the per-layer sums alone.
  step     measure, select, pack of the persisted layers into a device buffer, snapshot commit.
  graph    the same step replayed as a CUDA graph, with its decision read back.
  adamw    the optimizer step that also takes the drift (lc_adamw_step_measure), and its select.
  save     a step whose persisted layers go to a pinned host store, until they are durable.
  restore  a recovery: the newest version of every layer from the host store back into the device tensors.

`lie` says how the tensors lie:
  own      every tensor on an allocation boundary, as torch.empty gives it: everything is aligned.
  views    every array kind is one flat buffer with the tensors back to back in it, as sharded trainers keep
           parameters, moments and snapshots: a tensor behind an odd-sized one starts off a 16-byte boundary.
  clones   the parameters and moments are such views, but the snapshots (for adamw: the gradients) are tensors of
           their own, as w.clone() and autograd make them: weights and references then start at different
           offsets from a 16-byte boundary.
`world` > 1 gives the contiguous shard of every tensor that rank `rank` holds; shards of a world size that does not
divide the tensors are odd-sized.  `units` "tensors" makes every tensor its own layer.  `every` n persists every
n-th layer of a step (0: none), through threshold multipliers, so that each pass does the same work.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2609_27193_gb300 as P
from paper_2609_27193_gb300 import _abi

ALIGN = 256                    # bytes: where torch's allocator starts a tensor, and the packed sections
TAU, FAR = 1e-3, 1e12          # a threshold, and a multiplier of it that no drift reaches
NEVER = 1 << 30                # staleness bound that no pass reaches
HP = dict(lr=1e-5, beta1=0.9, beta2=0.95, eps=1e-8, weight_decay=0.1)
FIRST = 1                      # step of a state's first pass

TINY = dict(blocks=4, d=256, ffn=1024, kv=256, vocab=8000, tied=True)
SMALL = dict(blocks=12, d=768, ffn=3072, kv=768, vocab=32000, tied=True)
B1 = dict(blocks=16, d=2048, ffn=8192, kv=512, vocab=128256, tied=True)
B8 = dict(blocks=32, d=4096, ffn=14336, kv=1024, vocab=128256, tied=False)
PLAIN = dict(lie="own", dtype="bf16", units="layers", world=1, rank=0, every=0, accumulate=False)


def _case(name, path, shape, **more):
    return dict(PLAIN, **shape, **dict(more, name=name, path=path))


def listed():
    return [
        # the decision for the smallest model of the tests: launches and the readback are all of it
        _case("decide 6M", "decide", TINY),
        # the paper's literal drift (against the weights of the step before), each tensor a unit of its own
        _case("decide 1.2B tensors accumulate", "decide", B1, units="tensors", accumulate=True),
        # the decision of the benchmark's model: the most bytes that one call reads
        _case("decide 8B", "decide", B8),
        # a rank of three, its shards views of a flat buffer and the snapshots cloned from them
        _case("decide 1.2B/3 clones", "decide", B1, lie="clones", world=3, rank=1),
        # the same sums for a program that owns all of the GPU's memory itself
        _case("sums 1.2B", "sums", B1),
        # a whole step of the smallest model, and of an ordinary one; a quarter to a third of the layers persisted
        _case("step 6M", "step", TINY, every=3),
        _case("step 1.2B", "step", B1, every=4),
        # a whole step of a rank of three, everything in flat buffers
        _case("step 1.2B/3 views", "step", B1, lie="views", world=3, rank=1, every=4),
        # fp32 training of a small model, the step as a graph
        _case("graph 138M f32", "graph", SMALL, dtype="f32", every=4),
        # the optimizer step of an ordinary model
        _case("adamw 1.2B", "adamw", B1),
        # to the host and back; the host link bounds both
        _case("save 138M", "save", SMALL, every=4),
        _case("restore 138M", "restore", SMALL),
    ]


#: parameters (on this rank) of the smallest and largest drawn model of a path
RANGE = {"decide": (1e6, 7.5e9), "sums": (1e6, 2e9), "step": (1e6, 1.3e9), "graph": (1e6, 1.3e9),
         "adamw": (1e6, 1.3e9), "save": (1e6, 1.5e8), "restore": (1e6, 1.5e8)}


def draw(rng):
    path = rng.choice(["decide", "decide", "sums", "step", "step", "graph", "adamw", "save", "restore"])
    lo, hi = RANGE[path]
    world = rng.choice([1, 1, 1, 2, 3, 8])
    size = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    blocks = max(1, min(32, int(round(math.exp(rng.uniform(math.log(2), math.log(32)))))))
    wide, narrow = rng.uniform(2.5, 4.0), rng.choice([1, 4, 8])
    d = math.sqrt(0.8 * size * world / blocks / (2 + 2 / narrow + 3 * wide))
    d = max(16, int(d / 64) * 64) if d >= 128 and rng.random() < 0.5 else max(16, int(d))
    dtype = "f32" if path == "adamw" else rng.choice(["bf16", "bf16", "f32"])
    if path == "decide" and dtype == "f32" and size > 3.5e9:
        dtype = "bf16"
    return dict(path=path, blocks=blocks, d=d, ffn=int(d * wide), kv=max(1, d // narrow),
                vocab=max(16, int(0.2 * size * world / d)), tied=True, lie=rng.choice(["own", "views", "clones"]),
                dtype=dtype, units=rng.choice(["layers", "layers", "tensors"]), world=world,
                rank=rng.randrange(world), every=0 if path in ("decide", "sums", "adamw", "restore")
                else rng.choice([1, 3, 4, 8]),
                accumulate=path == "adamw" or (path in ("decide", "step") and rng.random() < 0.25))


# ---------------------------------------------------------------------------
# layout
# ---------------------------------------------------------------------------

def _tensors(c):
    """[(layer, numel)] of this rank's shard of every tensor, and the number of layers."""
    d, f, kv = c["d"], c["ffn"], c["kv"]
    groups = [[c["vocab"] * d]]
    groups += [[d * d, kv * d, kv * d, d * d, f * d, f * d, d * f, d, d]] * c["blocks"]
    groups += [[d]]
    if not c["tied"]:
        groups.append([c["vocab"] * d])
    out, layer = [], 0
    w, r = c["world"], c["rank"]
    for g in groups:
        for n in g:
            out.append((layer, max(1, n * (r + 1) // w - n * r // w)))
            layer += c["units"] == "tensors"
        layer += c["units"] != "tensors"
    return out, layer


def _moments(c):
    return c["path"] not in ("decide", "sums")


def _esz(c):
    return 4 if c["dtype"] == "f32" or c["path"] == "adamw" else 2


def _offsets(numels, esz, own):
    """Element offset of every tensor in a flat buffer, and the buffer's elements."""
    step, at, out = ALIGN // esz if own else 1, 0, []
    for n in numels:
        out.append(at)
        at = -(-(at + n) // step) * step
    return out, max(at, 1)


def _persisted(c, nlayers):
    return [c["path"] == "restore" or (c["every"] > 0 and l % c["every"] == 0) for l in range(nlayers)]


def _inputs(c, seed):
    """The training state a step finds: flat buffers and the tensors' views of them."""
    ts, nlayers = _tensors(c)
    numels = [n for _, n in ts]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    wt = torch.float32 if _esz(c) == 4 else torch.bfloat16
    own = c["lie"] == "own"
    flat, view = {}, {}

    def buffer(kind, dtype, aligned):   # zeros, so that the gaps between tensors are the same for everybody
        offs, n = _offsets(numels, torch.empty(0, dtype=dtype).element_size(), aligned)
        flat[kind] = torch.zeros(n, dtype=dtype, device=dev)
        view[kind] = [flat[kind][o:o + k] for o, k in zip(offs, numels)]

    adamw = c["path"] == "adamw"
    buffer("w", wt, own)
    if adamw:
        buffer("grad", torch.bfloat16, c["lie"] != "views")
        buffer("model", torch.bfloat16, own)
    else:
        buffer("r", wt, c["lie"] != "views")
    if _moments(c):
        buffer("m", torch.float32, own)
        buffer("v", torch.float32, own)
    drift = np.random.default_rng(seed).uniform(math.log(1e-5), math.log(1e-2), nlayers)
    for k, (layer, n) in enumerate(ts):
        x = torch.empty(n, dtype=torch.float32, device=dev).normal_(0.0, 0.02, generator=g)
        if adamw:
            view["w"][k].copy_(x)
            view["grad"][k].copy_(x.normal_(0.0, 1e-3, generator=g))
        else:
            view["r"][k].copy_(x)
            y = torch.empty(n, dtype=torch.float32, device=dev).normal_(0.0, 0.02, generator=g)
            view["w"][k].copy_(x.add_(y, alpha=math.exp(drift[layer])))
            del y
        del x
        if _moments(c):
            view["m"][k].normal_(0.0, 1e-3, generator=g)
            view["v"][k].normal_(0.0, 1e-6, generator=g).abs_()
    return ts, nlayers, flat, view


def prepare(case, seed):
    c = dict(case)
    ts, nlayers, flat, view = _inputs(c, seed)
    none = [None] * len(ts)
    segs = [P.segment(layer, w, r, m, v) for (layer, _), w, r, m, v in
            zip(ts, view["w"], view.get("r", none), view.get("m", none), view.get("v", none))]
    s = dict(case=c, flat=flat, view=view, t=FIRST, nlayers=nlayers)
    if c["path"] == "sums":
        s["segs"] = (_abi.lc_segment * len(segs))(*segs)
        s["keep"] = segs
        s["sums"] = torch.zeros(3 * nlayers, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return s
    lc = P.LayerCheck(mode=P.LC_DRIFT_ACCUMULATE if c["accumulate"] or c["path"] == "adamw" else P.LC_DRIFT_SNAPSHOT)
    sel = _persisted(c, nlayers)
    lc.register_layout(segs, nlayers, [0.0 if x else FAR for x in sel])
    s["lc"] = lc
    if c["path"] == "adamw":
        lc.register_optimizer(view["grad"], view["model"])
    stream_bytes = sum(lc.layer_block_bytes(l) for l in range(nlayers) if sel[l])
    if c["path"] in ("step", "graph"):
        s["dst"] = torch.zeros(max(16, stream_bytes), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    if c["path"] == "graph":
        lc.step_graph_create(TAU, NEVER, s["dst"])
    if c["path"] in ("save", "restore"):
        blocks = [-(-lc.layer_block_bytes(l) // 4096) * 4096 for l in range(nlayers)]
        s["store"] = P.Store(lc, capacity_bytes=sum(blocks) + 2 * sum(set(blocks)) + (1 << 20), versions_per_layer=1)
    if c["path"] == "restore":
        lc.measure(s["t"])
        lc.select(TAU, NEVER)
        lc.pack_async(s["store"])
        lc.commit_snapshot()
        lc.wait_durable(s["t"])
        for kind in ("w", "r", "m", "v"):      # what the failure destroyed
            flat[kind].zero_()
    torch.cuda.synchronize()
    return s


def _bits(x):
    """A float tensor's bits, for outputs that are copies."""
    return x.view(torch.int16 if x.element_size() == 2 else torch.int32)


def _newest(store):
    """The block of the version persisted last, as the store holds it; the array keeps the store."""
    v = store.version(len(store) - 1)
    block = (ctypes.c_int64 * (v["bytes"] // 8)).from_address(v["host_ptr"])
    block.store = store
    return np.frombuffer(block, dtype=np.int64)


def run(s):
    c, t, flat = s["case"], s["t"], s["flat"]
    path = c["path"]
    if path == "sums":
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)   # calls of one device go in order
        _abi.check(P.library().lc_measure_noalloc(0, stream, s["segs"], len(s["segs"]), s["nlayers"],
                                                  ctypes.c_void_p(s["sums"].data_ptr())))
        return dict(sums=s["sums"])
    lc = s["lc"]
    if path == "restore":
        steps = lc.restore(s["store"], t)
        return dict(steps=steps, w=_bits(flat["w"]), r=_bits(flat["r"]), m=_bits(flat["m"]), v=_bits(flat["v"]))
    s["t"] = t + 1
    if path == "graph":
        mask, u, nbytes = lc.step_wait(lc.step_graph_launch())
    else:
        if path == "adamw":
            lc.adamw_step_measure(t, **HP)
        else:
            lc.measure(t)
        mask, u, nbytes = lc.select(TAU, NEVER)
    out = dict(mask=mask, u=u, nbytes=nbytes)
    if path == "adamw":
        out.update(w=flat["w"], m=flat["m"], v=flat["v"], model=_bits(flat["model"]))
        return out
    if path == "step":
        lc.pack_device(s["dst"])
        lc.commit_snapshot()
    if path == "save":
        lc.pack_async(s["store"])
        lc.commit_snapshot()
        lc.wait_durable(t)
    if path in ("step", "graph"):
        out["stream"] = s["dst"][:nbytes].view(torch.int64)
    if path in ("step", "graph", "save") or c["accumulate"]:
        out["r"] = _bits(flat["r"])
    if path == "save":
        out["block"] = _newest(s["store"])
    return out


# ---------------------------------------------------------------------------
# floors, tolerances, 64-bit results
# ---------------------------------------------------------------------------

def work(case):
    c = dict(case)
    ts, nlayers = _tensors(c)
    sel, e = _persisted(c, nlayers), _esz(c)
    n = sum(k for _, k in ts)
    p = sum(k for l, k in ts if sel[l])
    if c["path"] == "adamw":       # w, m, v and the gradient in; w, m, v and the model copy out
        return dict(bytes=n * (12 + 2 + 12 + 2), flops=16 * n)
    if c["path"] == "restore":     # a block in; w, r, m and v out
        return dict(bytes=p * (e + 8 + 2 * e + 8), flops=0)
    # w and r in; of a persisted layer the moments in, the stream and the reference out
    b = 2 * e * n + p * (8 + e + 8 + e)
    if c["accumulate"]:
        b += e * (n - p)
    return dict(bytes=b, flops=4 * n)


def tolerance(case):
    c = dict(case)
    if c["path"] == "restore":
        return "exact"
    if c["path"] == "adamw":       # one rounding to 24 bits for each operation of the step: 4.4e-8 off exact()
        return dict(rel=2e-7)
    # 24-bit chains of at most 32 terms, joined in 64 bits: off exact() by up to 1.8e-9 from fp32 weights, and by
    # up to 5e-11 from bf16 ones, whose differences leave most of the 24 bits unused
    return dict(rel=1e-8 if _esz(c) == 4 else 1e-9)


def _sums64(view, k, w="w", r="r"):
    d = a = 0.0
    x, y = view[w][k], view[r][k]
    for i in range(0, x.numel(), 1 << 28):
        p, q = x[i:i + (1 << 28)].double(), y[i:i + (1 << 28)].double()
        a += float(q.abs().sum())
        d += float(p.sub_(q).abs_().sum())
    return d, a


def exact(case, seed):
    """The drift of every layer (and the updated optimizer state) in 64 bits; copies have none."""
    c = dict(case)
    if c["path"] == "restore":
        return None
    ts, nlayers, flat, view = _inputs(c, seed)
    sums = np.zeros((nlayers, 3))
    done = {}
    if c["path"] == "adamw":
        for kind in ("w", "m", "v"):
            done[kind] = torch.zeros(flat[kind].numel(), dtype=torch.float64, device="cuda")
        offs, _ = _offsets([n for _, n in ts], 4, c["lie"] == "own")
    for k, (layer, n) in enumerate(ts):
        if c["path"] == "adamw":
            g, w = view["grad"][k].double(), view["w"][k].double()
            m = HP["beta1"] * view["m"][k].double() + (1 - HP["beta1"]) * g
            v = HP["beta2"] * view["v"][k].double() + (1 - HP["beta2"]) * g * g
            del g
            new = w * (1 - HP["lr"] * HP["weight_decay"])
            new -= HP["lr"] / (1 - HP["beta1"] ** FIRST) * m / ((v / (1 - HP["beta2"] ** FIRST)).sqrt_() + HP["eps"])
            for kind, x in (("w", new), ("m", m), ("v", v)):
                done[kind][offs[k]:offs[k] + n] = x
            # the drift is that of the stored weights: the update is far below their last place
            d = a = None
            del m, v, new, w
        else:
            d, a = _sums64(view, k)
            sums[layer] += (d, a, n)
    if c["path"] == "sums":
        return dict(sums=sums.reshape(-1))
    out = dict(mask=None, nbytes=None)
    if c["path"] == "adamw":
        return dict(out, u=None, model=None, **done)
    u = (sums[:, 0] / sums[:, 2]) / (sums[:, 1] / sums[:, 2] + 1e-8)
    return dict(out, u=u, stream=None, r=None, block=None)
