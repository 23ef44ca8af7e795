"""The performance cases: what users of the FMM have it do, through the public Python API.

Four shapes of call:
  step      a time step of an N-body code: the tree is rebuilt over moved points, then evaluated;
  eval      one evaluation on a tree built earlier (an iterative solver on fixed points);
  diff      the potentials and the backward pass of torch.autograd with respect to densities and points;
  adaptive  one evaluation over an adaptive tree set up earlier.
The operators (`precompute`) are made once per program and belong to `prepare`.

Point families: uniform in the unit cube, uniform on the unit sphere, and the mixed cloud (half
uniform, half on a small sphere inside the cube) that adaptive refinement is for.
"""
import math

import torch

import paper_2604_19243_gb300 as fmmlib

CUBE = ((0.0, 0.0, 0.0), 1.0)
BALL = ((-1.0, -1.0, -1.0), 2.0)
INV4PI = 1.0 / (4.0 * math.pi)


def _case(name, call, dist, n, p, depth, precision="fp16x3", outputs="both", charge="u01", kernel="laplace", kappa=0.0,
          m2l="dense", capacity=0):
    c = dict(call=call, dist=dist, n=n, p=p, depth=depth, precision=precision, outputs=outputs, charge=charge,
             kernel=kernel, kappa=kappa, m2l=m2l, capacity=capacity)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the small plain case: default precision, potentials only; launches and host work count
        _case("step_cube20k_p4_fp32", "step", "cube", 20_000, 4, 3, precision="fp32", outputs="phi"),
        # a middle-sized particle code that needs forces only, on a ragged number of points
        _case("step_sphere150k_force", "step", "sphere", 150_001, 6, 5, outputs="grad"),
        # a million particles of both signs: the ordinary time step
        _case("step_cube1m_p6", "step", "cube", 1_048_576, 6, 5, charge="u11"),
        # the headline: 8.39M points on a sphere, tree build and potentials and gradients
        _case("step_sphere8m_p6", "step", "sphere", 8_388_608, 6, 7),
        # the differentiation case: forward and backward through torch.autograd
        _case("diff_cube262k_p6", "diff", "cube", 262_144, 6, 4, charge="normal"),
        # the default precision (plain FP32) on a fixed tree
        _case("eval_cube1m_p6_fp32", "eval", "cube", 1_048_576, 6, 5, precision="fp32", charge="u11"),
        # high order: p = 8 with 16 points per leaf
        _case("eval_cube4m_p8", "eval", "cube", 4_194_304, 8, 6),
        # high order with the FFT form of the M2L
        _case("eval_cube524k_p8_fft", "eval", "cube", 524_288, 8, 5, precision="fp32", m2l="fft"),
        # screened interactions on fixed points: one operator set per level
        _case("eval_cube1m_yukawa", "eval", "cube", 1_000_003, 6, 5, kernel="yukawa", kappa=10.0, charge="u11"),
        # scattering: complex densities on a closed surface
        _case("eval_sphere131k_helmholtz", "eval", "sphere", 131_072, 5, 4, kernel="helmholtz", kappa=2.0, charge="u11"),
        # a strongly non-uniform cloud over an adaptive tree
        _case("adaptive_mixed1m_p6_fp32", "adaptive", "mixed", 1_048_576, 6, 9, precision="fp32", capacity=64),
        # double precision, as used to validate the others
        _case("eval_cube100k_p6_fp64", "eval", "cube", 100_003, 6, 4, precision="fp64", charge="u11"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _depth(dist, n, ppl):
    """The depth whose non-empty leaves hold about ppl points."""
    per = 8.0 if dist != "sphere" else 4.0
    boxes = n / ppl / (1.0 if dist != "sphere" else 4.56)
    return max(2, min(8, round(math.log(max(boxes, 1.0)) / math.log(per))))


def _draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "diff", "eval", "eval", "fft", "yukawa", "helmholtz", "adaptive", "fp64"])
    dist = rng.choice(["cube", "sphere"])
    charge = rng.choice(["u01", "u11", "normal"])
    outputs = rng.choice(["both", "both", "grad", "phi"])
    ppl = math.exp(rng.uniform(math.log(12.0), math.log(140.0)))
    if kind in ("step", "eval"):
        precision = rng.choice(["fp16x3"] * 4 + ["fp32"] * 2 + ["bf16x6", "tf32x3"])
        p = rng.choice([4, 5, 6, 6, 6, 8])
        n = _logint(rng, 2_000, 8_300_000 if p <= 6 and precision == "fp16x3" else 1_500_000)
        return _case("", kind, dist, n, p, _depth(dist, n, ppl), precision, outputs, charge)
    if kind == "diff":
        n = _logint(rng, 2_000, 1_000_000)
        return _case("", "diff", dist, n, rng.choice([4, 6]), _depth(dist, n, ppl), rng.choice(["fp16x3", "fp16x3", "fp32"]), charge=charge)
    if kind == "fft":
        n = _logint(rng, 4_000, 1_000_000)
        return _case("", "eval", dist, n, rng.choice([4, 6, 8]), _depth(dist, n, ppl), "fp32", outputs, charge, m2l="fft")
    if kind == "yukawa":
        n = _logint(rng, 4_000, 1_500_000)
        return _case("", rng.choice(["step", "eval"]), dist, n, rng.choice([4, 6]), min(5, _depth(dist, n, ppl)), outputs=outputs,
                     charge=charge, kernel="yukawa", kappa=rng.choice([1.0, 3.0, 10.0]))
    if kind == "helmholtz":
        n = _logint(rng, 4_000, 300_000)
        return _case("", rng.choice(["step", "eval"]), dist, n, rng.choice([4, 5]), min(5, _depth(dist, n, ppl)), outputs=outputs,
                     charge=charge, kernel="helmholtz", kappa=rng.choice([1.0, 2.0, 3.0]))
    if kind == "adaptive":
        n = _logint(rng, 10_000, 1_000_000)
        return _case("", "adaptive", "mixed", n, rng.choice([4, 6]), min(9, 2 + _depth("cube", n, 48.0)), "fp32", outputs, charge,
                     capacity=rng.randint(24, 96))
    n = _logint(rng, 4_000, 130_000)
    return _case("", rng.choice(["step", "eval"]), dist, n, rng.choice([4, 6]), _depth(dist, n, ppl), "fp64", outputs, charge)


def _cost(case):
    w = work(case)
    # FP64 and the plain FP32 arithmetic run far below the tensor cores' rate
    rate = {"fp64": 0.8e12, "fp32": 2.0e13}.get(case["precision"], 1.0e14)
    return max(w["bytes"] / 5e12, w["flops"] / rate)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


def _points(case, g, dt):
    n = case["n"]
    if case["dist"] == "cube":
        return torch.rand(n, 3, generator=g, device="cuda", dtype=dt)
    if case["dist"] == "sphere":
        v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
        return (v / v.norm(dim=1, keepdim=True)).to(dt)
    v = torch.randn(n - n // 2, 3, generator=g, device="cuda", dtype=torch.float64)
    v = 0.5 + 0.15 * v / v.norm(dim=1, keepdim=True)
    return torch.cat([torch.rand(n // 2, 3, generator=g, device="cuda", dtype=dt), v.to(dt)])


def _charges(kind, n, g, dt):
    if kind == "normal":
        return torch.randn(n, generator=g, device="cuda", dtype=dt)
    q = torch.rand(n, generator=g, device="cuda", dtype=dt)
    return 2 * q - 1 if kind == "u11" else q


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    x = _points(case, g, dt)
    q = _charges(case["charge"], case["n"], g, dt)
    if case["kernel"] == "helmholtz":
        q = torch.complex(q, _charges(case["charge"], case["n"], g, dt))
    w = torch.randn(case["n"], generator=g, device="cuda", dtype=dt) if case["call"] == "diff" else None
    return x, q, w


def prepare(case, seed):
    x, q, w = _inputs(case, seed)
    f = fmmlib.FMM(p=case["p"], depth=case["depth"], precision=case["precision"],
                   domain=BALL if case["dist"] == "sphere" else CUBE, kernel=case["kernel"], kappa=case["kappa"],
                   m2l=case["m2l"])
    f.precompute()
    if case["call"] != "step":
        f.build_tree(x)
    if case["call"] == "adaptive":
        f.adaptive_setup(case["capacity"])
    if case["call"] == "diff":
        q.requires_grad_()
        x.requires_grad_()
    return {"case": case, "fmm": f, "x": x, "q": q, "w": w}


def run(state):
    c, f, x, q = state["case"], state["fmm"], state["x"], state["q"]
    if c["call"] == "diff":
        phi = fmmlib.FmmFunction.apply(q, x, f)
        dq, dx = torch.autograd.grad(phi, (q, x), state["w"])
        return {"phi": phi.detach(), "dq": dq, "dx": dx}
    if c["call"] == "step":
        f.build_tree(x)
    evaluate = f.adaptive_evaluate if c["call"] == "adaptive" else f.evaluate
    phi, grad = evaluate(q, gradient=c["outputs"] != "phi", potential=c["outputs"] != "grad")
    return {"phi": phi, "grad": grad}


def _tree_counts(case):
    """(near-field pairs, non-empty boxes of the levels 2..depth, V-list entries), expected values of the family."""
    n, d = case["n"], case["depth"]
    if case["dist"] == "sphere":   # 4.56 * 4^l boxes meet the unit sphere; 15.2 neighbours, 44 V entries each
        boxes = [min(n, 4.56 * 4 ** lev) for lev in range(2, d + 1)]
        return 15.2 * n * max(1.0, n / boxes[-1]), sum(boxes), 44.0 * sum(boxes)
    if case["dist"] == "mixed":    # leaves between capacity / 8 and capacity points
        leaves = n / max(1.0, 0.28 * case["capacity"])
        return 15.2 * n * 0.28 * case["capacity"], 1.2 * leaves, 1.2 * leaves * 60.0
    pairs = boxes = entries = 0.0
    for lev in range(2, d + 1):
        m = 2 ** lev
        b = min(float(n), float(m) ** 3)
        u, c = ((3 * m - 2) / m) ** 3, 8 * ((3 * (m // 2) - 2) / (m // 2)) ** 3
        fill = min(1.0, n / float(m) ** 3)
        boxes += b
        entries += b * (c - u) * fill
        pairs = n * max(1.0, u * n / float(m) ** 3)
    return pairs, boxes, entries


def work(case):
    n, ns = case["n"], 6 * (case["p"] - 1) ** 2 + 2
    es = 8 if case["precision"] == "fp64" else 4
    cx = 2 if case["kernel"] == "helmholtz" else 1
    pairs, boxes, entries = _tree_counts(case)
    per_pair = {"laplace": 20, "yukawa": 27, "helmholtz": 45}[case["kernel"]]
    k = ns * cx
    per_entry = 8.0 * (2 * case["p"]) ** 2 * (case["p"] + 1) if case["m2l"] == "fft" else 2.0 * k * k
    outs = {"both": 4, "grad": 3, "phi": 1}[case["outputs"]]
    flops = pairs * per_pair + 2 * n * ns * per_pair + entries * per_entry + boxes * 4 * 2.0 * k * k
    nbytes = n * es * (3 + cx + outs * cx)
    if case["call"] == "diff":     # the field of the densities, the transposed map and the field of the cotangents
        flops, nbytes = 3 * flops, n * es * (3 + 1 + 1 + 1 + 1 + 3)
    return {"bytes": float(nbytes), "flops": float(flops)}


def _direct(x, q, case, want_phi, want_grad):
    """The sums of every pair in 64 bits."""
    x = x.double().detach()
    q = q.detach().to(torch.complex128 if q.is_complex() else torch.float64)
    n, kappa = x.shape[0], case["kappa"]
    phi, grad = torch.empty(n, dtype=q.dtype, device=x.device), torch.empty(n, 3, dtype=q.dtype, device=x.device)
    chunk = max(1, (1 << 26) // n)
    ax = [x[:, a].contiguous() for a in range(3)]
    for i in range(0, n, chunk):
        j = min(n, i + chunk)
        d = [ax[a][i:j, None] - ax[a][None, :] for a in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        ri = torch.where(r2 > 0, r2.rsqrt(), torch.zeros((), dtype=r2.dtype, device=r2.device))
        if case["kernel"] == "laplace":
            w, dw = ri, -ri * ri * ri
        else:
            r = r2 * ri
            if case["kernel"] == "yukawa":
                w = ri * torch.exp(-kappa * r)
                dw = -w * (1 + kappa * r) * ri * ri
            else:
                w = ri * torch.complex(torch.cos(kappa * r), torch.sin(kappa * r))
                dw = w * torch.complex(-torch.ones_like(r), kappa * r) * (ri * ri)
        if want_phi:
            phi[i:j] = w @ q
        if want_grad:
            for a in range(3):
                grad[i:j, a] = (dw * d[a]) @ q
    return phi * INV4PI if want_phi else None, grad * INV4PI if want_grad else None


def exact(case, seed):
    if case["n"] > (140_000 if case["kernel"] == "helmholtz" else 280_000):
        return None
    x, q, w = _inputs(case, seed)
    if case["call"] == "diff":
        phi, grad = _direct(x, q, case, True, True)
        psi, grad_w = _direct(x, w, case, True, True)   # the kernel is symmetric
        return {"phi": phi, "dq": psi, "dx": w.double()[:, None] * grad + q.double()[:, None] * grad_w}
    phi, grad = _direct(x, q, case, case["outputs"] != "grad", case["outputs"] != "phi")
    return {"phi": phi, "grad": grad}
