"""The work a user has this library do, as cases that can be timed and compared.

Each case is one pass through the public entry points of `paper_2512_18345_gb300.binding`:
CKKS operations on ciphertexts (HMult and rescale, rotations, hoisted rotations, linear
transforms), batched plans, and the stage calls from which callers compose pipelines of
their own.  Ring degrees are the two the library supports (2^12 and 2^16); the other sizes
are those of `inputs.WORKLOADS`, the tests and the benchmark, and ragged ones between them.

A case holds plain values:
  kind            which calls a pass makes (see `run`)
  logn, L, K, dnum, bits   the context's parameters
  level           ciphertext level (limbs) the calls work at
  tc              tensor-core base conversion (else CUDA cores)
  and per kind: n (rotations of a hoisted set, items of a plan), lo / hi / mix (levels and
  operations of a plan), baby / giant (dense transform), levels / which (radix level of
  CoeffToSlot).

All outputs are residues, that is whole numbers, so `exact` has nothing to add: they have to
stay equal, bit for bit.
"""
import math

import torch

from paper_2512_18345_gb300 import binding, inputs

_L24 = dict(logn=16, L=24, K=8, dnum=3, bits=31, tc=True)
_L48 = dict(logn=16, L=48, K=12, dnum=4, bits=31, tc=True)


def listed():
    return [
        # the smallest call: HMult, relinearisation and rescale on the small ring (leveled
        # circuits of a few products); launches and latency count
        dict(name="hmult_rescale_small", kind="hmult_rescale", logn=12, L=4, K=2, dnum=2, bits=30, level=4, tc=False),
        # one CoeffToSlot level on the small ring: many small stages in one call
        dict(name="transform_small", kind="transform_dh", logn=12, L=8, K=2, dnum=4, bits=30, level=8, tc=True,
             levels=3, which=1),
        # one rotation, the call an application makes between other work
        dict(name="rotate_L24", kind="rotate", level=24, **_L24),
        # a product late in a circuit: low odd level, last digit partial, the default conversion
        dict(name="hmult_rescale_low", kind="hmult_rescale", level=11, **{**_L24, "tc": False}),
        # key switching alone at a ragged level of the paper's alpha = 12 parameters
        dict(name="keyswitch_L24_a12", kind="keyswitch", logn=16, L=24, K=12, dnum=2, bits=31, level=23, tc=True),
        # the rotations of one ciphertext that a convolution or a matrix product needs
        dict(name="hoisted_L24", kind="hoisted", level=24, n=8, **_L24),
        # the benchmark's step: eight rotations with eight keys, one captured plan
        dict(name="batch8_rotate", kind="batch", level=24, n=8, lo=24, hi=24, mix=0, **_L24),
        # a server's mixed load: 64 rotations and relinearisations at levels 4..24
        dict(name="batch64_mixed", kind="batch", level=24, n=64, lo=4, hi=24, mix=20251222, **_L24),
        # a dense matrix-vector product (16 x 8 baby and giant steps)
        dict(name="bsgs_L24", kind="transform", level=24, baby=16, giant=8, **_L24),
        # one CoeffToSlot level of bootstrapping at the paper's parameters, the largest call
        dict(name="cts_level_L48", kind="transform_dh", level=48, levels=3, which=1, **_L48),
        # stage calls composed by the caller: decompose a polynomial, bring one down, at an odd level
        dict(name="stages_l17", kind="stages", level=17, **_L24),
        # plaintext product, sum and rescale: a weighted sum without key switching
        dict(name="pmult_add_rescale", kind="pmult_add_rescale", level=24, **_L24),
    ]


_KINDS = ("hmult_rescale", "rotate", "keyswitch", "hoisted", "batch", "transform", "transform_dh", "stages",
          "pmult_add_rescale")


def _between(rng, lo, hi):
    """A whole number in [lo, hi], even over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(_KINDS)
    c = dict(kind=kind, logn=rng.choice((12, 16, 16)), bits=rng.choice((30, 31, 31)), tc=rng.random() < 0.7)
    c["L"] = _between(rng, 3, 48 if kind in ("rotate", "keyswitch", "hmult_rescale", "stages", "transform_dh") else 30)
    # digits of at most 12 limbs (the tensor-core conversion's limit), at most four of them
    c["dnum"] = rng.randint(max(1, -(-c["L"] // 12)), min(4, c["L"]))
    alpha = -(-c["L"] // c["dnum"])
    c["K"] = rng.randint(max(1, alpha - 1), min(12, alpha + 1))
    c["level"] = rng.randint(max(2, c["L"] // 3), c["L"])
    if kind == "hoisted":
        c["n"] = _between(rng, 2, 12)
    elif kind == "batch":
        c["n"] = _between(rng, 1, 24)
        c["hi"] = c["level"]
        c["lo"] = rng.randint(1, c["level"])
        c["mix"] = rng.randint(1, 1 << 30)
    elif kind == "transform":
        c["baby"], c["giant"] = _between(rng, 2, 16), _between(rng, 1, 6)
    elif kind == "transform_dh":
        c["levels"] = rng.randint(3, 4)
        c["which"] = rng.randrange(c["levels"])
    return c


# ------------------------------------------------------------------ what a case consists of

def _params(case):
    return inputs.make_params(1 << case["logn"], case["L"], case["K"], case["dnum"], case["bits"])


def _items(case):
    """(operation, level, rotation) of a plan's items: rotations at one level, or a mix."""
    n, slots = case["n"], 1 << (case["logn"] - 1)
    if not case["mix"]:
        return [("rotate", case["hi"], 1 + (i * 4093) % (slots - 1)) for i in range(n)]
    items = inputs.batch_items(inputs.rng(case["mix"]), n, case["lo"], case["hi"])
    return [(i["op"], i["level"], 1 + i["rot"] % (slots - 1)) for i in items]


def _bsgs(case):
    return inputs.transform_plans(1 << case["logn"], case["levels"], "cts")[case["which"]]


class _Draws:
    """Uniform residues (what ciphertexts, keys and encoded plaintexts look like) on the GPU."""

    def __init__(self, P, seed):
        self.P = P
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def residues(self, primes, *lead):
        q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
        out = torch.empty(*lead, len(primes), self.P.N, dtype=torch.int32, device="cuda")
        for row in out.view(-1, len(primes), self.P.N):
            row.copy_(torch.randint(0, 1 << 62, row.shape, generator=self.g, device="cuda").remainder_(q))
        return out

    def poly(self, level, *lead):
        return self.residues(self.P.q[:level], *lead)

    def key(self):
        return self.residues(self.P.primes, self.P.dnum, 2)


def prepare(case, seed):
    P = _params(case)
    d, level, kind = _Draws(P, seed), case["level"], case["kind"]
    ctx = binding.Context.from_params(P)
    ctx.set_bconv(binding.FHE_BCONV_TC if case["tc"] else binding.FHE_BCONV_SCALAR)
    s = dict(case=case, ctx=ctx)

    def rot_keys(rots):
        for r in rots:
            ctx.set_rot_key(r, d.key())

    if kind == "hmult_rescale":
        ctx.set_relin_key(d.key())
        s["a"], s["b"] = d.poly(level, 2), d.poly(level, 2)
    elif kind == "rotate":
        rot_keys([5])
        s["a"] = d.poly(level, 2)
    elif kind == "keyswitch":
        ctx.set_relin_key(d.key())
        s["a"] = d.poly(level)
    elif kind == "hoisted":
        s["rots"] = [1 << i for i in range(case["n"])] if case["n"] < case["logn"] else list(range(1, case["n"] + 1))
        rot_keys(s["rots"])
        s["a"] = d.poly(level, 2)
    elif kind == "batch":
        items = _items(case)
        rot_keys(sorted({r for op, _, r in items if op == "rotate"}))
        ctx.set_relin_key(d.key())
        plan = []
        for op, l, r in items:
            it = dict(op=binding.FHE_OP_ROTATE if op == "rotate" else binding.FHE_OP_RELIN, level=l, rot=r)
            it["in"] = d.poly(l, 2)
            if op != "rotate":
                it["in2"] = d.poly(l, 2)
            it["out"] = torch.zeros_like(it["in"])
            plan.append(it)
        s["outs"] = [it["out"] for it in plan]
        s["plan"] = ctx.batch_plan(plan, binding.FHE_PLAN_GRAPH)
    elif kind == "transform":
        rot_keys(sorted(set(range(1, case["baby"])) | {case["baby"] * g for g in range(1, case["giant"])}))
        s["a"], s["diags"] = d.poly(level, 2), d.poly(level, case["baby"] * case["giant"])
    elif kind == "transform_dh":
        s["t"] = _bsgs(case)
        rot_keys(s["t"].rotations())
        s["a"] = d.poly(level, 2)
        s["diags"] = d.residues(P.q[:level] + P.p, s["t"].n_diag)
    elif kind == "stages":
        s["a"], s["u"] = d.poly(level), d.residues(P.q[:level] + P.p)
    elif kind == "pmult_add_rescale":
        s["a"], s["b"], s["pt"] = d.poly(level, 2), d.poly(level, 2), d.poly(level)
    else:
        raise ValueError(kind)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind, level = case["kind"], case["level"]
    if kind == "hmult_rescale":
        return ctx.rescale(ctx.hmult(s["a"], s["b"], level), level)
    if kind == "rotate":
        return ctx.rotate(s["a"], level, 5)
    if kind == "keyswitch":
        return ctx.keyswitch(s["a"], level)
    if kind == "hoisted":
        return ctx.rotate_hoisted(s["a"], level, s["rots"])
    if kind == "batch":
        s["plan"].launch()
        return s["outs"]
    if kind == "transform":
        return ctx.linear_transform(s["a"], level, s["diags"], case["baby"], case["giant"])
    if kind == "transform_dh":
        return ctx.linear_transform_dh(s["a"], level, s["t"].baby, s["t"].giant, s["diags"], s["t"].idx)
    if kind == "stages":
        return ctx.modup(s["a"], level), ctx.moddown(s["u"], level)
    x = ctx.pmult(s["a"], s["pt"], level)
    return ctx.rescale(ctx.add(x, s["b"], level), level)


def exact(case, seed):
    return None  # whole numbers throughout: equality is asked of them, not closeness


# ------------------------------------------------------------------ what a pass cannot do without

def _add(*parts):
    return tuple(sum(x) for x in zip(*parts))


def _times(n, part):
    return tuple(n * x for x in part)


def work(case):
    """Bytes: inputs, keys and outputs once each (no intermediate).  flops: modular
    multiplications, additions and subtractions (3 a butterfly, 2 a multiply-accumulate)."""
    P = _params(case)
    N, K, kind, l = P.N, P.K, case["kind"], case["level"]
    limb = 4.0 * N
    ntt = (0.0, 1.5 * N * case["logn"])  # one limb's transform

    def digits(l):
        return [min(l, lo + P.alpha) - lo for lo in range(0, l, P.alpha)]

    def key(l):
        return (len(digits(l)) * 2 * (l + K) * limb, 0.0)

    def modup(l):
        conv = sum(n * (l + K - n) for n in digits(l))
        return _add(_times(len(digits(l)) * (l + K), ntt), (0.0, 2.0 * N * conv))

    def inner(l):
        return (0.0, 4.0 * N * len(digits(l)) * (l + K))

    def moddown(l, n=2):
        return _times(n, _add(_times(K + l, ntt), (0.0, 2.0 * N * (K * l + l))))

    def switch(l):
        return _add(modup(l), inner(l), moddown(l))

    def io(limbs):
        return (limbs * limb, 0.0)

    def rescale(l):
        return _times(2 * l, _add(ntt, (0.0, 2.0 * N)))

    if kind == "hmult_rescale":
        parts = [io(4 * l + 2 * (l - 1)), key(l), (0.0, 7.0 * N * l), switch(l), rescale(l)]
    elif kind == "rotate":
        parts = [io(4 * l), key(l), switch(l)]
    elif kind == "keyswitch":
        parts = [io(3 * l), key(l), switch(l)]
    elif kind == "hoisted":
        n = case["n"]
        parts = [io(2 * l + 2 * n * l), _times(n, key(l)), modup(l), _times(n, _add(inner(l), moddown(l)))]
    elif kind == "batch":
        items = _items(case)
        relins = [lv for op, lv, _ in items if op != "rotate"]
        rots = {}
        for op, lv, r in items:
            if op == "rotate":
                rots[r] = max(lv, rots.get(r, 0))
        parts = [_add(io((4 if op == "rotate" else 6) * lv), switch(lv)) for op, lv, _ in items]
        parts += [key(lv) for lv in rots.values()] + ([key(max(relins))] if relins else [])
    elif kind == "transform":
        b, g = case["baby"], case["giant"]
        keys = len(set(range(1, b)) | {b * x for x in range(1, g)})
        parts = [io(4 * l + b * g * l), _times(keys, key(l)), (0.0, 4.0 * N * l * b * g), modup(l),
                 _times(b - 1, _add(inner(l), moddown(l))), _times(g - 1, switch(l))]
    elif kind == "transform_dh":
        t = _bsgs(case)
        nb, ng = sum(1 for r in t.baby if r), sum(1 for r in t.giant if r)
        parts = [io(4 * l + t.n_diag * (l + K)), _times(len(t.rotations()), key(l)),
                 (0.0, 4.0 * N * (l + K) * t.n_diag), modup(l), _times(nb, inner(l)),
                 _times(ng, _add(moddown(l, 1), modup(l), inner(l))), moddown(l)]
    elif kind == "stages":
        parts = [io(l + len(digits(l)) * (l + K) + 2 * l + K), modup(l), moddown(l, 1)]
    else:
        parts = [io(5 * l + 2 * (l - 1)), (0.0, 4.0 * N * l), rescale(l)]
    total = _add(*parts)
    return {"bytes": total[0], "flops": total[1]}
