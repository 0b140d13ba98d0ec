"""The work that a program using the DensityKV bank library has it do, as cases to time and compare.

Three kinds of call, all through the Python binding of the C ABI:

  attend   dkv_bank_attend: a block's queries over [bank | local window], the call that every
           denoising pass of every block makes;
  update   dkv_bank_admit (or admit_rope) and dkv_bank_compress: a finalized block offered to the
           banks, once per generated block;
  step     both, in the order of a generation loop;
  order    dkv_candidate_order_noalloc: scores and order of one head for hosts that cannot allocate.

Banks are in their steady state (full, or filled to a stated share of the budget) with keys from
recurring clusters, as a rollout leaves them; blocks mix recurring and fresh clusters.  An update's
state holds several different blocks and each pass offers the next, so the bank goes on as it does in
a rollout.  Inputs are drawn with torch on the device of the bank.
"""
import math
import random

import torch

from paper_2608_27922_gb300 import dkv

CLUSTERS, KAPPA, FRESH, BLOCKS = 64, 20.0, 8, 4

_BASE = dict(kind="update", H=12, d=128, dtype="bf16", mode="tensor", N=4680, M=9360, fill=1.0, mixed=False,
             layer_heads=0, sync=True, order="score", evict="mandatory_densest", desc="k", rope="off", p=2,
             Nq=0, W=0)


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest whole step: 2 heads of 64 dimensions in fp32, 256-token blocks, 512-token banks.  Latency and
        # launches count; small models, unit tests and exactness checks of a port run this.
        _case(name="tiny_fp32_step", kind="step", H=2, d=64, dtype="fp32", mode="fp32", N=256, M=512, Nq=256, W=256),
        # One Wan-1.3B-shaped layer: a 3-frame block's queries over a full 6-frame bank and a 3-frame window.
        _case(name="layer_attend", kind="attend", Nq=4680, W=4680),
        # The same layer denoising one frame at a time early in a video: 1,560 queries, a bank that is not yet full
        # and ends inside a tile, the sink frame and four recent frames as the window.
        _case(name="frame_attend", kind="attend", Nq=1560, W=7800, fill=0.741),
        # Four layers of the Wan-14B-shaped stack in one handle (40 heads each, budgets from an eighth to the whole
        # of 18,720): what one call of a whole-model step does, at a tenth of its heads.
        _case(name="stack_attend", kind="attend", H=160, M=18720, mixed=True, layer_heads=40, Nq=4680, W=4680),
        # The Wan-1.3B-shaped layer's update at the end of each block, bank full: every candidate scored and ordered,
        # the densest states evicted, the block admitted.
        _case(name="layer_update"),
        # The update of those four stacked layers with budgets of their own, one call for all.
        _case(name="stack_update", H=160, M=18720, mixed=True, layer_heads=40),
        # A long video's bank of 21 frames (32,760 states a head).
        _case(name="large_bank_update", M=32760),
        # One frame offered with its temporal rotation still on (re-zeroed on the way in), a budget that ends inside a
        # tile.
        _case(name="frame_update_rope", N=1560, M=9001, rope="interleaved"),
        # The [K; V] retention descriptor with a prefix of its own in each head (two ablations that users switch on).
        _case(name="layer_update_kv", desc="kv", sync=False),
        # The exactness mode on bf16 banks: direct fp32 differences, for runs that must reproduce retained sets.
        _case(name="exact_update", mode="fp32", N=1560),
        # Attention of an fp32 bank (fp32 models, and references for the bf16 path).
        _case(name="fp32_attend", kind="attend", dtype="fp32", mode="fp32", M=4680, Nq=1560, W=1560),
        # Scores and order of one head without device allocation.
        _case(name="order_noalloc", kind="order", H=1, mode="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        r = rng.random()
        if r < 0.35:
            c = _case(kind="attend", H=_log(rng, 1, 160), M=_log(rng, 256, 32760), Nq=_log(rng, 16, 4680),
                      W=rng.choice([0, _log(rng, 64, 9360), _log(rng, 64, 9360)]), N=256)
        elif r < 0.7:
            c = _case(H=_log(rng, 1, 160), M=_log(rng, 256, 32760), N=_log(rng, 64, 4680),
                      rope=rng.choice(["off", "off", "interleaved", "half"]), desc=rng.choice(["k", "k", "k", "kv"]),
                      sync=rng.random() < 0.7, p=rng.choice([2, 2, 2, 1, 4]),
                      order=rng.choice(["score", "score", "score", "source"]),
                      evict=rng.choice(["mandatory_densest", "mandatory_densest", "densest", "mandatory_source"]))
        elif r < 0.8:
            c = _case(kind="step", H=_log(rng, 1, 12), d=rng.choice([64, 128]), dtype=rng.choice(["fp32", "bf16"]),
                      mode="fp32", N=_log(rng, 32, 512), M=_log(rng, 64, 1024), Nq=_log(rng, 32, 512),
                      W=_log(rng, 32, 512))
        elif r < 0.87:
            c = _case(H=_log(rng, 1, 12), d=rng.choice([64, 128]), dtype=rng.choice(["fp32", "bf16"]), mode="fp32",
                      N=_log(rng, 64, 4680), M=_log(rng, 256, 9360), desc=rng.choice(["k", "k", "k", "kv"]))
        elif r < 0.94:
            c = _case(kind="attend", H=_log(rng, 1, 12), d=rng.choice([64, 128]), dtype=rng.choice(["fp32", "bf16"]),
                      mode="fp32", M=_log(rng, 256, 9360), Nq=_log(rng, 16, 4680), W=_log(rng, 64, 4680), N=256)
        else:
            c = _case(kind="order", H=1, d=rng.choice([64, 128]), dtype=rng.choice(["fp32", "bf16"]), mode="fp32",
                      N=_log(rng, 64, 16384), M=_log(rng, 64, 32760))
        c["fill"] = rng.choice([1.0, 1.0, round(rng.uniform(0.3, 0.99), 3)])
        c["mixed"] = c["kind"] in ("attend", "update") and c["H"] >= 8 and rng.random() < 0.3
        if c["kind"] == "update" and c["H"] % 4 == 0 and rng.random() < 0.5:
            c["layer_heads"] = c["H"] // 4
        if _cost(c) <= top:
            return c


# ---------------------------------------------------------------- sizes and work
def _budgets(c):
    if not c["mixed"]:
        return [c["M"]] * c["H"]
    r = random.Random(c["M"] + 1000003 * c["H"])
    b = [max(1, c["M"] >> r.randrange(4)) for _ in range(c["H"])]
    b[0] = c["M"]
    return b


def _occupancy(c):
    return [max(1, min(b, int(round(c["fill"] * b)))) for b in _budgets(c)]


def _attend_work(c):
    es = 2 if c["dtype"] == "bf16" else 4
    keys = sum(_occupancy(c)) + c["H"] * c["W"]
    return (2 * keys + 2 * c["H"] * c["Nq"]) * c["d"] * es, 4 * c["Nq"] * keys * c["d"]


def _update_work(c):
    """Scores of every candidate against the bank, the growth of every bank state along the candidates
    (whose order is known only once the scores are), survivors against the evicted and the admitted
    against the new bank, for a prefix that admits the whole block (or the smallest budget)."""
    es = 2 if c["dtype"] == "bf16" else 4
    occ, bud = _occupancy(c), _budgets(c)
    lh = c["layer_heads"] or c["H"]
    flops = nbytes = 0
    for l in range(0, c["H"], lh):
        r = min(c["N"], min(bud[l:l + lh]))
        for m, M in zip(occ[l:l + lh], bud[l:l + lh]):
            e = max(0, m + r - M)
            pairs = (c["N"] * m if c["order"] == "score" else 0) + m * r + (m - e) * e + r * (m + r - e)
            flops += 2 * c["d"] * (2 if c["desc"] == "kv" else 1) * pairs
            # keys of the bank and of the block in, densities in and out, admitted keys and values moved
            nbytes += (m + c["N"]) * c["d"] * es + 4 * r * c["d"] * es + 16 * m + 32 * r
    return nbytes, flops


def work(c):
    b = f = 0
    if c["kind"] in ("attend", "step"):
        x = _attend_work(c)
        b, f = b + x[0], f + x[1]
    if c["kind"] in ("update", "step"):
        x = _update_work(c)
        b, f = b + x[0], f + x[1]
    if c["kind"] == "order":
        es = 2 if c["dtype"] == "bf16" else 4
        m = _occupancy(c)[0]
        b, f = (m + c["N"]) * c["d"] * es + 4 * m + 8 * c["N"], 2 * c["d"] * m * c["N"]
    return {"bytes": b, "flops": f}


def _cost(c):
    """About the seconds of a pass: matrix units for the tensor mode, fp32 units for the exactness mode."""
    w = work(c)
    return w["flops"] / (1e15 if c["mode"] == "tensor" else 1.5e13) + w["bytes"] / 5e12


# ---------------------------------------------------------------- inputs
def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


class _Source:
    """Keys around per-head cluster centres on the sphere of radius sqrt(d), spread as a von Mises-Fisher
    mixture of concentration KAPPA a dimension; values N(0, 1)."""

    def __init__(self, c, seed):
        self.c, self.gen = c, torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        n = CLUSTERS + FRESH * BLOCKS
        mu = torch.randn(c["H"], n, c["d"], generator=self.gen, device="cuda")
        self.mu = mu / mu.norm(dim=-1, keepdim=True)

    def keys(self, n, fresh=None, share=0.0):
        H, d, g = self.c["H"], self.c["d"], self.gen
        which = torch.randint(0, CLUSTERS, (H, n), generator=g, device="cuda")
        if fresh is not None:
            new = CLUSTERS + FRESH * fresh + torch.randint(0, FRESH, (H, n), generator=g, device="cuda")
            which = torch.where(torch.rand(H, n, generator=g, device="cuda") < share, new, which)
        out = torch.empty(H, n, d, device="cuda", dtype=_dtype(self.c))
        for h in range(0, H, 32):
            x = torch.randn(out[h:h + 32].shape, generator=g, device="cuda").mul_(1.0 / math.sqrt(KAPPA * (d - 1)))
            x += torch.gather(self.mu[h:h + 32], 1, which[h:h + 32, :, None].expand(-1, -1, d))
            out[h:h + 32] = x * (math.sqrt(d) / x.norm(dim=-1, keepdim=True))
        return out

    def values(self, n):
        out = torch.empty(self.c["H"], n, self.c["d"], device="cuda", dtype=_dtype(self.c))
        for h in range(0, out.shape[0], 32):
            out[h:h + 32] = torch.randn(out[h:h + 32].shape, generator=self.gen, device="cuda")
        return out


def _sigma2(c):
    return c["d"] / 2.0 * (2 if c["desc"] == "kv" else 1)


def _pair_w(c, a, b, va, vb):
    """Soft-Riesz interactions of rows a and b (and their values, for the [K; V] descriptor)."""
    if c["desc"] == "kv":
        a, b = torch.cat([a, va], -1), torch.cat([b, vb], -1)
    d2 = (a * a).sum(-1)[:, None] + (b * b).sum(-1)[None, :] - 2.0 * (a @ b.T)
    return (1.0 + d2.clamp_(min=0.0) / _sigma2(c)) ** -c["p"]


def _rotate(k, t, theta, layout, sign):
    """k rotated by sign * t * theta in each rotation pair, in float64."""
    ang = sign * t.double()[:, None] * theta.double()[None, :]
    co, si = ang.cos(), ang.sin()
    k = k.double()
    half = k.shape[-1] // 2
    x, y = (k[..., 0::2], k[..., 1::2]) if layout == "interleaved" else (k[..., :half], k[..., half:])
    u, v = x * co - y * si, x * si + y * co
    return torch.stack([u, v], -1).flatten(-2) if layout == "interleaved" else torch.cat([u, v], -1)


def _inputs(c, seed):
    s = _Source(c, seed)
    occ = _occupancy(c)
    x = {"occ": occ, "k": s.keys(max(occ)), "v": s.values(max(occ))}
    H, m, p = c["H"], max(occ), c["p"]
    if c["kind"] != "attend":
        # densities of the retained set (fp32 is enough for an input), and baselines that they have grown from
        # or shrunk below by the factors that a rollout's banks hold
        rho = torch.zeros(H, m, device="cuda")
        for h in range(H):
            k, v = x["k"][h, :occ[h]].float(), x["v"][h, :occ[h]].float()
            for r in range(0, occ[h], 4096):
                rho[h, r:min(r + 4096, occ[h])] = _pair_w(c, k[r:r + 4096], k, v[r:r + 4096], v).sum(1) - 1.0
        grown = torch.empty(H, m, device="cuda").uniform_(0.7, 1.5, generator=s.gen)
        x["rho"], x["base"] = rho, torch.clamp(rho / grown, min=1e-6)
        x["blocks"] = []
        for b in range(1 if c["kind"] == "order" else BLOCKS):
            k, v = s.keys(c["N"], fresh=b, share=0.4), s.values(c["N"])
            t = theta = None
            if c["rope"] != "off":
                n = c["d"] // 2 // 3
                theta = torch.zeros(c["d"] // 2, device="cuda")
                theta[:n] = 10000.0 ** (-torch.arange(n, device="cuda", dtype=torch.float64) / n)
                t = (3 * b + 7 + torch.arange(c["N"], device="cuda") * 3 // c["N"]).to(torch.int32)
                for h in range(H):
                    k[h] = _rotate(k[h], t, theta, c["rope"], 1.0)
            x["blocks"].append((k, v, t, theta))
    if c["Nq"]:
        x["q"] = s.keys(c["Nq"], fresh=0, share=0.4)
        x["kw"], x["vw"] = (s.keys(c["W"], fresh=0, share=0.4), s.values(c["W"])) if c["W"] else (None, None)
    return x


def _owned(bank, view):
    """The library's view of its workspace as a slice of the workspace tensor, which keeps it alive."""
    at = view.data_ptr() - bank.workspace.data_ptr()
    return bank.workspace[at:at + view.numel() * view.element_size()].view(view.dtype).view(view.shape)


def prepare(c, seed):
    x = _inputs(c, seed)
    state = {"case": c, "x": x, "t": 0}
    if c["kind"] == "order":
        state["params"] = dkv.dkv_params_default(c["d"])
        state["dtype"] = dkv.DKV_DTYPE_BF16 if c["dtype"] == "bf16" else dkv.DKV_DTYPE_FP32
        state["scores"] = torch.zeros(c["N"], device="cuda")
        state["perm"] = torch.zeros(c["N"], dtype=torch.int32, device="cuda")
        return state
    bank = dkv.BankLayer(c["H"], c["d"], _budgets(c), c["N"], _dtype(c), p=float(c["p"]), sync_heads=int(c["sync"]),
                         layer_heads=c["layer_heads"],
                         sigma=math.sqrt(_sigma2(c)),
                         score_mode=dkv.DKV_SCORE_TENSOR if c["mode"] == "tensor" else dkv.DKV_SCORE_FP32,
                         order=dkv.DKV_ORDER_SCORE if c["order"] == "score" else dkv.DKV_ORDER_SOURCE,
                         eviction={"mandatory_densest": dkv.DKV_EVICT_MANDATORY_DENSEST,
                                   "densest": dkv.DKV_EVICT_DENSEST,
                                   "mandatory_source": dkv.DKV_EVICT_MANDATORY_SOURCE}[c["evict"]],
                         descriptor=dkv.DKV_DESC_KV if c["desc"] == "kv" else dkv.DKV_DESC_K)
    occ, m = x["occ"], max(x["occ"])
    live = torch.arange(m, device="cuda")[None, :] < torch.tensor(occ, device="cuda")[:, None]
    bank.k[:, :m] = torch.where(live[..., None], x.pop("k"), 0)
    bank.v[:, :m] = torch.where(live[..., None], x.pop("v"), 0)
    if c["kind"] != "attend":
        bank.rho[:, :m], bank.base[:, :m] = x.pop("rho") * live, x.pop("base") * live
    else:
        bank.base[:, :m] = live
    bank.prov_step[:, :m] = torch.where(live, torch.arange(m, device="cuda")[None, :] // c["N"], -1)
    bank.prov_src[:, :m] = torch.where(live, torch.arange(m, device="cuda")[None, :] % c["N"], -1).to(torch.int32)
    bank.import_state(occ)
    state["bank"] = bank
    state["t0"] = m // c["N"] + 1
    if c["kind"] != "attend":
        mid = bank.intermediates()
        state["mid"] = {"perm": _owned(bank, mid["perm"])}
        if c["order"] == "score":
            state["mid"]["score"] = _owned(bank, mid["score"])
    return state


def _bits(t):
    """The same memory as whole numbers: keys and values are moved bit for bit."""
    return t.view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


def run(state):
    c, x = state["case"], state["x"]
    if c["kind"] == "order":
        k, _, _, _ = x["blocks"][0]
        dkv.dkv_candidate_order_noalloc(x["k"][0], x["base"][0], x["occ"][0], k[0], c["N"], c["d"], state["dtype"],
                                        state["params"], state["scores"], state["perm"])
        return {"score": state["scores"], "perm": state["perm"]}
    bank, out = state["bank"], {}
    if c["kind"] in ("attend", "step"):
        out["O"] = bank.attend(x["q"], x["kw"], x["vw"])
    if c["kind"] in ("update", "step"):
        k, v, t, theta = x["blocks"][state["t"] % BLOCKS]
        step = state["t0"] + state["t"]
        state["t"] += 1
        if t is None:
            bank.update(k, v, step)
        else:
            bank.update(k, v, step, t_coord=t, theta=theta,
                        rope_layout=dkv.DKV_ROPE_INTERLEAVED if c["rope"] == "interleaved" else dkv.DKV_ROPE_HALF)
        out.update(state["mid"])
        out.update(k=_bits(bank.k), v=_bits(bank.v), rho=bank.rho, base=bank.base, knorm=bank.knorm,
                   prov_step=bank.prov_step, prov_src=bank.prov_src, occupancy=bank.occupancy)
    return out


def tolerance(c):
    if c["kind"] == "attend":
        return {"rel": 1e-2, "max": 0.2} if c["mode"] == "tensor" or c["dtype"] == "bf16" else {"rel": 1e-5}
    if c["mode"] == "tensor":
        # With the bank columns of the score pass added in another order, candidates whose scores lie closer than
        # their rounding change places, and with them the slots that they enter: whole rows, measured as rel 0.0035,
        # max 0.25 and 0.0053 of the whole values.  The scores themselves are 1.3e-7 off float64.
        return {"rel": 0.015, "max": 0.9, "differ": 0.01}
    # fp32 decisions are the same in any correct version that sums in the documented order
    return {"rel": 1e-2, "max": 0.2} if c["kind"] == "step" and c["dtype"] == "bf16" else {"rel": 1e-5}


# ---------------------------------------------------------------- the same in 64 bits
def _exact_score(c, k, v, base, bk, bv):
    """Mean of w / b over the bank for each row of k."""
    k, v, bk, bv = k.double(), v.double(), bk.double(), bv.double()
    inv = 1.0 / base.double()
    out = torch.empty(k.shape[0], dtype=torch.float64, device="cuda")
    for r in range(0, k.shape[0], 2048):
        out[r:r + 2048] = _pair_w(c, k[r:r + 2048], bk, v[r:r + 2048], bv) @ inv / bk.shape[0]
    return out


def exact(c, seed):
    """Attention outputs and candidate scores in float64.  What an update leaves in the bank has no such value here:
    which slot holds which state follows from the order of scores that can lie closer than their rounding."""
    w = work(c)
    if w["flops"] > 1.2e13:
        return None
    x = _inputs(c, seed)
    occ, out = x["occ"], {}
    if c["kind"] == "order":
        k, v, _, _ = x["blocks"][0]
        m = occ[0]
        return {"score": _exact_score(c, k[0], v[0], x["base"][0, :m], x["k"][0, :m], x["v"][0, :m]), "perm": None}
    if c["kind"] in ("attend", "step"):
        o = torch.empty(x["q"].shape, dtype=torch.float64, device="cuda")
        for h in range(c["H"]):
            k, v = x["k"][h, :occ[h]], x["v"][h, :occ[h]]
            if c["W"]:
                k, v = torch.cat([k, x["kw"][h]]), torch.cat([v, x["vw"][h]])
            k, v = k.double(), v.double()
            for r in range(0, c["Nq"], 1024):
                s = x["q"][h, r:r + 1024].double() @ k.T / math.sqrt(c["d"])
                o[h, r:r + 1024] = torch.softmax(s, -1) @ v
        out["O"] = o
    if c["kind"] in ("update", "step") and c["order"] == "score":
        k, v, t, theta = x["blocks"][0]
        s = torch.empty(c["H"], c["N"], dtype=torch.float64, device="cuda")
        for h in range(c["H"]):
            kh = k[h] if t is None else _rotate(k[h], t, theta, c["rope"], -1.0).to(k.dtype)
            s[h] = _exact_score(c, kh, v[h], x["base"][h, :occ[h]], x["k"][h, :occ[h]], x["v"][h, :occ[h]])
        out["score"] = s
    return out
