"""Timed cases: what users of this library have it do, through its public entry points.

Every case is one call (or the short sequence of calls) that a program makes: a
whole solve from device arrays, a solve from host arrays, a product with new
charges on a kept plan, a batch of problems, the plain FP64 method, the direct
sum that measures errors, the learned selector's plan and its training step.
Sizes, degrees, leaf sizes and distributions are those of the workloads
(workloads.py), the benchmark and the tests, or odd sizes between them.

Potentials of an FP32_BULK plan are single-precision results (1e-7 to 1e-6 by
the option's definition: FP32 kernel evaluations) that the library hands over
in float64 arrays; the programs that ask for that option keep them in float32,
and so do these cases.  FP64 plans' potentials stay float64.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2012_06925_gb300 import binding as B

EXACT_PAIRS = 1.2e11          # the 64-bit direct sum of more pairs would take too long
KERNELS = {"coulomb": B.COULOMB, "yukawa": B.YUKAWA, "oscillatory": B.OSCILLATORY,
           "reg_coulomb": B.REG_COULOMB}
DEGREES = (3, 4, 5, 6, 7, 8)  # the learned selector's degree set


def listed():
    return [
        # the smallest solve: a molecule-sized problem, where launches and
        # synchronisations count (the batched workload's smallest problem)
        dict(name="small_solve", what="solve", kind="uniform", M=1000, N=0, kernel="coulomb", kappa=0.0,
             n=6, theta=0.7, leaf=500, fp64=False),
        # an iterative solver's product on a kept plan: new charges, then the
        # captured compute phase (boundary elements on a sphere)
        dict(name="matvec_sphere", what="matvec", kind="sphere", M=20011, N=0, kernel="coulomb", kappa=0.0,
             n=6, theta=0.7, leaf=500, fp64=False),
        # ordinary solve with the wave kernel (kappa = pi), a clustered set
        dict(name="wave_plummer", what="solve", kind="plummer", M=100003, N=0, kernel="oscillatory",
             kappa=math.pi, n=6, theta=0.7, leaf=1000, fp64=False),
        # the benchmark's workload: 1E6 points, set-up and compute
        dict(name="uniform_1e6", what="solve", kind="uniform", M=1000000, N=0, kernel="coulomb", kappa=0.0,
             n=8, theta=0.7, leaf=2000, fp64=False),
        # the largest: targets and sources apart, screened kernel
        dict(name="unequal_yukawa", what="solve", kind="uniform", M=10000000, N=5000000, kernel="yukawa",
             kappa=0.5, n=7, theta=0.8, leaf=2000, fp64=False),
        # many independent problems of 1E3 to 1E5 points in one plan
        dict(name="batched_512", what="batch", count=512, nmin=1000, nmax=100000, n=6, theta=0.7, leaf=500,
             fp64=False),
        # softened gravity from host arrays, copies in and out included
        dict(name="host_softened", what="host", kind="plummer", M=300007, N=0, kernel="reg_coulomb",
             kappa=0.005, n=8, theta=0.7, leaf=2000, fp64=False),
        # the learned selector's multi-degree plan
        dict(name="learned_1e6", what="learned", kind="uniform", M=1000000, N=0, kernel="coulomb", kappa=0.0,
             n=8, theta=0.7, leaf=2000, fp64=False),
        # the plain FP64 method: the 2E4 workload, and an ordinary size
        dict(name="plain_fp64_2e4", what="solve", kind="uniform", M=20000, N=0, kernel="coulomb", kappa=0.0,
             n=4, theta=0.7, leaf=500, fp64=True),
        dict(name="fp64_yukawa_6e4", what="solve", kind="uniform", M=60013, N=50021, kernel="yukawa",
             kappa=0.5, n=7, theta=0.8, leaf=1000, fp64=True),
        # error measurement: the FP64 direct sum on sampled targets
        dict(name="direct_sampled", what="direct", kind="uniform", M=2000, N=1000000, kernel="coulomb",
             kappa=0.0),
        # one step of the selector's training (forward, backward, update)
        dict(name="train_step", what="train", batch=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    what = rng.choice(("solve", "solve", "solve", "unequal", "matvec", "batch", "host", "learned", "fp64", "fp64",
                       "direct", "train"))
    kind = rng.choice(("uniform", "sphere", "plummer", "gaussian"))
    kernel = rng.choice(("coulomb", "coulomb", "yukawa", "oscillatory", "reg_coulomb"))
    kappa = {"coulomb": 0.0, "yukawa": round(rng.uniform(0.1, 2.0), 3), "oscillatory": math.pi,
             "reg_coulomb": 0.005}[kernel]
    common = dict(kind=kind, kernel=kernel, kappa=kappa, n=rng.randint(4, 8),
                  theta=round(rng.uniform(0.6, 0.8), 3), leaf=rng.choice((500, 777, 1000, 2000)), fp64=False)
    fast = kernel in ("coulomb", "yukawa")
    if what == "solve":
        return dict(what="solve", M=_log(rng, 1e3, 1.2e6 if fast else 3e5), N=0, **common)
    if what == "unequal":
        return dict(what="solve", M=_log(rng, 1e4, 3e6 if fast else 3e5), N=_log(rng, 1e4, 1e6 if fast else 3e5),
                    **common)
    if what == "matvec":
        return dict(what="matvec", M=_log(rng, 2e3, 2e5), N=0, **common)
    if what == "batch":
        return dict(what="batch", count=rng.randint(8, 96), nmin=1000, nmax=_log(rng, 2e3, 4e4),
                    n=rng.randint(4, 7), theta=common["theta"], leaf=rng.choice((300, 500)), fp64=False)
    if what == "host":
        return dict(what="host", M=_log(rng, 2e3, 5e5 if fast else 2e5), N=0, **common)
    if what == "learned":
        common.update(kernel="coulomb", kappa=0.0, n=8, leaf=2000, theta=0.7, kind="uniform")
        return dict(what="learned", M=_log(rng, 1e5, 1e6), N=0, **common)
    if what == "fp64":
        common.update(fp64=True)
        return dict(what="solve", M=_log(rng, 2e3, 6e4), N=0, **common)
    if what == "direct":
        return dict(what="direct", kind=kind, M=_log(rng, 100, 5e3), N=_log(rng, 1e4, 6e5), kernel=kernel,
                    kappa=kappa)
    return dict(what="train", batch=rng.randint(200, 4096))


# ---- inputs ---------------------------------------------------------------------
def _points(kind, m, g):
    """(3, m) float64 points on the device, as workloads.py's distributions."""
    if kind == "uniform":
        return torch.rand(3, m, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    x = torch.randn(3, m, generator=g, device="cuda", dtype=torch.float64)
    if kind == "gaussian":
        return x * math.sqrt(3.0)
    x = x / x.norm(dim=0, keepdim=True).clamp_min(1e-300)
    if kind == "sphere":
        return x
    a, mmax = 0.1, 1.0 / (1.0 + 0.01) ** 1.5          # Plummer: scale radius 0.1, cut at 1
    u = (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * mmax).clamp_min(1e-12)
    return (x * (a / (u ** (-2.0 / 3.0) - 1.0).sqrt())).contiguous()


def _charges(m, g):
    return torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * 2 - 1


def _sizes(case):
    """Problem sizes of a batch: log-uniform quantiles, in a fixed shuffled order."""
    c, lo, hi = case["count"], math.log(case["nmin"]), math.log(case["nmax"])
    sizes = [int(round(math.exp(lo + (hi - lo) * (i + 0.5) / c))) for i in range(c)]
    random.Random(4).shuffle(sizes)
    return sizes


def _selector():
    """A multi-degree selector with an a-priori rule: degree d is taken where
    (r_t + r_s)/R is at most 0.75^(9/(d+1)) (equal error estimates), inside a
    box of clusters of up to 4E5 particles, as the trained one's."""
    parts = []
    for o, i in ((64, 6), (64, 64), (64, 64), (3 * len(DEGREES), 64)):
        w, b = np.zeros((o, i), np.float32), np.zeros(o, np.float32)
        if o == 64:
            w[0, 4 if i == 6 else 0] = 1.0
        else:
            w[:, 0] = 6.0
            for k, d in enumerate(DEGREES):
                b[3 * k:3 * k + 3] = -6.25 - 6.0 * 0.75 ** (9.0 / (d + 1))
        parts += [w.ravel(), b]
    lo = np.zeros(6, np.float32)
    hi = np.array([1.17, 1.17, 1.0, 1.0, 0.85, 1.0], np.float32)
    return B.Selector(DEGREES, np.concatenate(parts), lo, hi, log10_budget=-6.25)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + 17)
    what = case["what"]
    s = dict(what=what)
    if what == "train":
        b, nout = case["batch"], 3 * len(DEGREES)
        lim = torch.tensor([1.2, 1.2, 0.5, 0.5, 0.95, 0.1], device="cuda")
        x = (torch.rand(b, 6, generator=g, device="cuda") * lim).contiguous()
        deg = torch.tensor(DEGREES, device="cuda", dtype=torch.float32).repeat_interleave(3)
        y = (deg + 1) * torch.log10(x[:, 4:5].clamp_min(0.05)) - 1.0
        y = (y + 0.2 * torch.randn(b, nout, generator=g, device="cuda")).clamp_min(-15.0).contiguous()
        mask = (torch.rand(b, nout, generator=g, device="cuda") < 0.98).float()
        parts = []
        for o, i in ((64, 6), (64, 64), (64, 64), (nout, 64)):
            parts.append(torch.randn(o * i, generator=g, device="cuda") * math.sqrt(2.0 / i))
            parts.append(torch.full((o,), -4.0 if o == nout else 0.0, device="cuda"))
        p = torch.cat(parts)
        s.update(x=x, y=y, mask=mask, nout=nout, p=p, m=torch.zeros_like(p), v=torch.zeros_like(p),
                 grads=torch.empty_like(p), loss=torch.empty(1, device="cuda"), step=0)
        return s
    if what == "batch":
        sizes = _sizes(case)
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        total = int(off[-1])
        pts = _points("uniform", total, g)
        odd = torch.zeros(total, dtype=torch.bool, device="cuda")
        for i in range(1, len(sizes), 2):            # odd problems lie on the unit sphere
            odd[int(off[i]):int(off[i + 1])] = True
        pts = torch.where(odd, _points("sphere", total, g), pts).contiguous()
        q = torch.randn(total, generator=g, device="cuda", dtype=torch.float64)
        r = random.Random(seed)
        kernels = [B.YUKAWA if (i // 2) % 2 else B.COULOMB for i in range(len(sizes))]
        kappas = [r.uniform(0.1, 2.0) if k == B.YUKAWA else 0.0 for k in kernels]
        s.update(pts=pts, q=q, off=off, kernels=kernels, kappas=kappas,
                 kw=dict(n=case["n"], theta=case["theta"], N0=case["leaf"], M0=case["leaf"]))
        return s
    M, N = case["M"], case["N"]
    tgt = _points(case["kind"], M, g)
    # the unequal sets' sources are a Plummer sphere, as the workload's
    src = _points("plummer" if what == "solve" else case["kind"], N, g) if N else tgt
    q = _charges(N or M, g)
    s.update(tgt=tgt, src=src, q=q)
    if what == "direct":
        s.update(kernel=KERNELS[case["kernel"]], kappa=case["kappa"])
        return s
    prec = B.FP64 if case["fp64"] else B.FP32_BULK
    kw = dict(kernel=KERNELS[case["kernel"]], kappa=case["kappa"], n=case["n"], theta=case["theta"],
              N0=case["leaf"], M0=case["leaf"], precision=prec)
    s.update(kw=kw, fp64=case["fp64"])
    if what == "host":
        host = [t.cpu().pin_memory().numpy() for t in (tgt, q)]
        return dict(what=what, tgt=host[0], q=host[1], kw=kw)
    if what == "learned":
        kw.pop("n")
        s.update(selector=_selector())
    if what == "matvec":
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            # the plan starts from charges of its own; each product brings new ones
            plan = B.Plan(tgt, src, torch.ones_like(q), stream=st, **kw)
            s.update(plan=plan, phi=torch.empty(M, dtype=torch.float64, device="cuda"), stream=st)
        torch.cuda.current_stream().wait_stream(st)
    return s


def run(s):
    what = s["what"]
    if what == "train":
        B.mlp_gradients(s["p"], s["nout"], s["x"], s["y"], s["mask"], grads=s["grads"], loss=s["loss"])
        s["step"] += 1
        B.mlp_adam(s["p"], s["m"], s["v"], s["grads"], s["step"], 2e-3)
        return dict(loss=s["loss"], grads=s["grads"], params=s["p"])
    if what == "direct":
        return B.direct_sum(s["tgt"], s["src"], s["q"], s["kernel"], s["kappa"])
    if what == "host":
        phi, _ = B.solve_host(s["tgt"], s["tgt"], s["q"], **s["kw"])
        return phi.astype(np.float32)
    if what == "matvec":
        st = s["stream"]
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            s["plan"].set_charges(s["q"])
            out = s["plan"].compute_graph(s["phi"], st).float()
        torch.cuda.current_stream().wait_stream(st)
        return out
    if what == "batch":
        with B.Plan.batch(s["pts"], s["off"], s["pts"], s["off"], s["q"], s["kernels"], s["kappas"],
                          **s["kw"]) as plan:
            return plan.compute().float()
    if what == "learned":
        with B.Plan.learned(s["tgt"], s["src"], s["q"], s["selector"], **s["kw"]) as plan:
            return plan.compute().float()
    with B.Plan(s["tgt"], s["src"], s["q"], **s["kw"]) as plan:
        phi = plan.compute()
        return phi if s["fp64"] else phi.float()


# ---- work and exact values ------------------------------------------------------
def _evaluations(m, n_src, n, leaf):
    """Kernel evaluations the method needs, roughly: every target meets the
    particles of about 50 leaves and about 38 proxy grids (theta 0.7), at most
    every source."""
    mean = float(n_src)
    while mean > leaf:
        mean /= 8.0
    return float(m) * min(float(n_src), 50.0 * mean + 38.0 * (n + 1) ** 3)


def work(case):
    what = case["what"]
    if what == "train":
        nw = 6 * 64 + 2 * 64 * 64 + 64 * 18 + 3 * 64 + 18
        b = case["batch"]
        return dict(bytes=4.0 * b * (6 + 2 * 18) + 4.0 * nw * 7, flops=6.0 * b * nw + 12.0 * nw)
    if what == "batch":
        sizes = _sizes(case)
        ev = sum(_evaluations(m, m, case["n"], case["leaf"]) for m in sizes)
        # half Coulomb (20 flops an evaluation), half Yukawa (28)
        return dict(bytes=(24.0 + 8.0 + 4.0) * sum(sizes), flops=24.0 * ev)
    m, n_src = case["M"], case["N"] or case["M"]
    flops = 20.0 if case["kernel"] in ("coulomb", "reg_coulomb") else 28.0
    nbytes = 24.0 * m + (24.0 * n_src if case["N"] else 0.0) + 8.0 * n_src
    if what == "direct":
        return dict(bytes=nbytes + 8.0 * m, flops=flops * m * n_src)
    if what == "matvec":                               # new charges in, potentials out, points in the plan
        nbytes = 24.0 * m + 8.0 * m
    return dict(bytes=nbytes + (8.0 if case["fp64"] else 4.0) * m,
                flops=flops * _evaluations(m, n_src, case["n"], case["leaf"]))


def _direct64(tgt, src, q, kernel, kappa):
    m, n_src = tgt.shape[1], src.shape[1]
    out = torch.empty(m, dtype=torch.float64, device=tgt.device)
    step = max(1, int(1.5e8) // n_src)
    for i in range(0, m, step):
        t = tgt[:, i:i + step]
        r2 = None
        for d in range(3):
            x = t[d][:, None] - src[d][None, :]
            r2 = x.mul_(x) if r2 is None else r2.addcmul_(x, x)
        zero = r2 == 0
        if kernel == B.REG_COULOMB:
            gr = (r2 + kappa * kappa).rsqrt_()
        else:
            r = r2.sqrt_()
            if kernel == B.YUKAWA:
                gr = torch.exp(r * -kappa).div_(r)
            elif kernel == B.OSCILLATORY:
                gr = torch.sin(r * kappa).div_(r)
            else:
                gr = r.reciprocal_()
        out[i:i + step] = gr.masked_fill_(zero, 0.0) @ q
    return out


def _exact_train(s):
    def rnd(t):                                        # the documented bf16 roundings
        return t.float().bfloat16().double()

    p, nout = s["p"].double(), s["nout"]
    ws, bs, o = [], [], 0
    for a, i in ((64, 6), (64, 64), (64, 64), (nout, 64)):
        ws.append(rnd(p[o:o + a * i]).view(a, i))
        o += a * i
        bs.append(p[o:o + a])
        o += a
    acts, zs = [rnd(s["x"])], []
    for k in range(3):
        zs.append(acts[-1] @ ws[k].T + bs[k])
        acts.append(rnd(zs[-1].clamp_min(0)))
    y = acts[-1] @ ws[3].T + bs[3]
    mask, diff = s["mask"].double(), y - s["y"].double()
    cnt = mask.sum().clamp_min(1.0)
    loss = ((mask * diff) ** 2).sum() / cnt
    gz, parts = 2.0 * mask * diff / cnt, []
    for k in (3, 2, 1, 0):
        parts = [(gz.T @ acts[k]).reshape(-1), gz.sum(0)] + parts
        if k:
            gz = (gz @ ws[k]) * (zs[k - 1] > 0)
    grads = torch.cat(parts)
    m, v = 0.1 * grads, 0.001 * grads * grads
    params = p - 2e-3 * (m / (1 - 0.9)) / ((v / (1 - 0.999)).sqrt() + 1e-8)
    return dict(loss=loss.reshape(1), grads=grads, params=params)


def exact(case, seed):
    what = case["what"]
    if what == "train":
        return _exact_train(prepare(case, seed))
    if what == "batch":
        sizes = _sizes(case)
        if sum(float(m) * m for m in sizes) > EXACT_PAIRS:
            return None
        s = prepare(case, seed)
        out = []
        for i, k in enumerate(s["kernels"]):
            a, b = int(s["off"][i]), int(s["off"][i + 1])
            out.append(_direct64(s["pts"][:, a:b], s["pts"][:, a:b], s["q"][a:b], k, s["kappas"][i]))
        return torch.cat(out)
    if float(case["M"]) * (case["N"] or case["M"]) > EXACT_PAIRS:
        return None
    s = prepare(case, seed)
    if what == "host":
        tgt, q = torch.from_numpy(s["tgt"]).cuda(), torch.from_numpy(s["q"]).cuda()
        return _direct64(tgt, tgt, q, s["kw"]["kernel"], s["kw"]["kappa"]).cpu().numpy()
    return _direct64(s["tgt"], s["src"], s["q"], KERNELS[case["kernel"]], case["kappa"])
