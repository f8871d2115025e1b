"""Performance cases of the layered-media FMM: what a program has it compute.

A case is one call (or the build and evaluation of one time step) of the public
Python interface, over the range of sizes, orders, media and forms the library
is used with:

* ``call = "step"``      new positions every time: ``build_device`` and
                         ``evaluate_device`` (potentials and fields);
* ``call = "evaluate"``  fixed positions, new charges: ``evaluate_device``;
* ``call = "product"``   the matrix-vector product of a Krylov solver on host
                         vectors: ``evaluate`` without fields;
* ``call = "batch"``     many independent problems: one batch evaluation.

``form`` is the arithmetic of the context ("f64" or "f32").  The float32 form
computes in float32 whatever the type of the arrays that carry its results, and
the program that chose it keeps its potentials and fields in float32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1908_10863_gb300 import LayeredFMM, workloads
from paper_1908_10863_gb300.lfmm import LayeredFMMBatch

MEDIA = {"config": workloads.EPS_CONFIG, "contrast": workloads.EPS_HIGH_CONTRAST, "paper": workloads.EPS_PAPER}


def _case(points, n, p, form, call, medium="config", nrhs=1, k=1, nmin=0):
    return {"points": points, "n": n, "p": p, "form": form, "call": call, "medium": medium, "nrhs": nrhs, "k": k,
            "nmin": nmin}


def listed():
    def named(name, *a, **kw):
        return dict(_case(*a, **kw), name=name)

    return [
        # the smallest problem, in double precision: 1,000 charges in the middle layer
        named("middle_1k_f64", "middle", 1000, 10, "f64", "step"),
        # the accuracy setting: irregular domains at the highest order (errors of 1e-10)
        named("domains_3k_p20_f64", "domains", 2848, 20, "f64", "step", medium="paper"),
        # the plain double precision method on an ordinary problem
        named("slabs_64k_f64", "slabs", 65536, 10, "f64", "step"),
        # one product of a small integral-equation solve (host vectors, potentials only)
        named("domains_3k_product_f32", "domains", 2848, 10, "f32", "product", medium="paper"),
        # the float32 form on an ordinary problem, positions moving every step
        named("slabs_64k_f32", "slabs", 65536, 10, "f32", "step"),
        # low order, fixed positions: fast approximate products
        named("slabs_262k_p6_f32", "slabs", 262144, 6, "f32", "evaluate"),
        # the float32 form at its highest order
        named("slabs_64k_p14_f32", "slabs", 65536, 14, "f32", "step"),
        # the headline problem: 1M charges in three layers
        named("slabs_1m_f32", "slabs", 1048576, 10, "f32", "step"),
        # every charge next to an interface: reaction pairs in the near field
        named("interfaces_50k_f32", "interfaces", 50001, 10, "f32", "step"),
        # a medium of four layers
        named("four_layers_262k_f32", "four", 262143, 10, "f32", "step", medium="four"),
        # 64 charge vectors over one geometry (block Krylov, many excitations)
        named("slabs_262k_64_vectors_f32", "slabs", 262144, 10, "f32", "evaluate", nrhs=64),
        # twelve uneven problems, 2,000 to 100,000 charges each, evaluated together
        named("batch_12_f32", "slabs", 100000, 10, "f32", "batch", k=12, nmin=2000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["f32", "f32", "f32", "f32_high", "f64", "f64", "f64_high", "interfaces", "interfaces_f64",
                       "four", "vectors", "batch", "product"])
    medium = rng.choice(["config", "config", "contrast", "paper"])
    points = rng.choice(["slabs", "slabs", "middle", "domains"])
    call = rng.choice(["step", "step", "evaluate"])
    if kind == "f32":
        return _case(points, _log(rng, 1000, 1048576), rng.randint(4, 10), "f32", call, medium)
    if kind == "f32_high":
        return _case(points, _log(rng, 1000, 65536), rng.randint(11, 14), "f32", call, medium)
    if kind == "f64":
        return _case(points, _log(rng, 1000, 65536), rng.randint(4, 10), "f64", call, medium)
    if kind == "f64_high":
        return _case(points, _log(rng, 1000, 3000), rng.choice([11, 12, 14, 16, 18, 20]), "f64", call, medium)
    if kind == "interfaces":
        return _case("interfaces", _log(rng, 4000, 131072), rng.randint(6, 10), "f32", call, medium)
    if kind == "interfaces_f64":
        return _case("interfaces", _log(rng, 1000, 3000), rng.randint(6, 10), "f64", call, medium)
    if kind == "four":
        return _case("four", _log(rng, 4000, 262144), rng.randint(6, 10), "f32", call, "four")
    if kind == "vectors":
        n = _log(rng, 4096, 262144)
        return _case("slabs", n, rng.randint(6, 10), rng.choice(["f32", "f32", "f64"]) if n < 8192 else "f32",
                     "evaluate", medium, nrhs=_log(rng, 2, 64) if n >= 8192 else _log(rng, 2, 16))
    if kind == "batch":
        return _case("slabs", _log(rng, 8000, 100000), rng.randint(6, 10), "f32", "batch", medium,
                     k=rng.randint(3, 12), nmin=2000)
    return _case(points, _log(rng, 1000, 20000), rng.randint(6, 12), rng.choice(["f32", "f32", "f64"]), "product",
                 medium)


def _sizes(case):
    """Charges of each problem: log-uniform from nmin to n, all odd sizes but the last."""
    k, n, lo = case["k"], case["n"], case["nmin"]
    if k == 1:
        return [n]
    return [int(round(lo * (n / lo) ** (i / (k - 1)))) | (1 if i < k - 1 else 0) for i in range(k)]


def _workload(case, n, seed):
    pts = case["points"]
    if pts == "four":
        return workloads.four_layers(n, seed=seed)
    if pts == "domains":  # the shares of the three domains are those of the paper's smallest run
        c0, c1 = n * 912 // 2848, n * 640 // 2848
        w = workloads.paper_p4((c0, c1, n - c0 - c1), seed=seed)
        w.eps = np.array(MEDIA[case["medium"]], dtype=np.float64)
        return w
    make = {"middle": workloads.config1, "slabs": workloads.config2, "interfaces": workloads.near_interface}[pts]
    return make(n, seed=seed, eps=MEDIA[case["medium"]])


def _problems(case, seed):
    return [_workload(case, n, seed * 64 + i) for i, n in enumerate(_sizes(case))]


def _charges(case, w, seed):
    """[n] or [nrhs, n] charges on the GPU, uniform in [-1, 1]."""
    if case["nrhs"] == 1:
        return torch.from_numpy(w.q).cuda()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.rand((case["nrhs"], w.n), dtype=torch.float64, device="cuda", generator=gen) * 2 - 1


def prepare(case, seed):
    single = case["form"] == "f32"
    ws = _problems(case, seed)
    fmms = [LayeredFMM(w.d, w.eps, case["p"], precision=1 if single else 0) for w in ws]
    st = {"call": case["call"], "single": single}
    if case["call"] == "product":
        fmms[0].build(ws[0].xyz, ws[0].layer)
        st.update(fmm=fmms[0], q=ws[0].q)
        return st
    xyz = [torch.from_numpy(w.xyz).cuda() for w in ws]
    layer = [torch.from_numpy(w.layer).cuda() for w in ws]
    if case["call"] != "step":
        for f, x, l in zip(fmms, xyz, layer):
            f.build_device(x, l)
    if case["call"] == "batch":
        q = torch.cat([torch.from_numpy(w.q).cuda() for w in ws])
        st.update(batch=LayeredFMMBatch(fmms), q=q, phi=torch.empty_like(q), field=q.new_empty(3 * q.numel()))
        return st
    q = _charges(case, ws[0], seed)
    st.update(fmm=fmms[0], xyz=xyz[0], layer=layer[0], q=q, phi=torch.empty_like(q),
              field=q.new_empty(tuple(q.shape) + (3,)))
    return st


def run(st):
    if st["call"] == "product":
        phi, _ = st["fmm"].evaluate(st["q"], field=False)
        return {"phi": phi.astype(np.float32) if st["single"] else phi}
    if st["call"] == "batch":
        st["batch"].evaluate_device(st["q"], st["phi"], st["field"])
    else:
        if st["call"] == "step":
            st["fmm"].build_device(st["xyz"], st["layer"])
        st["fmm"].evaluate_device(st["q"], st["phi"], st["field"])
    if st["single"]:
        return {"phi": st["phi"].float(), "field": st["field"].float()}
    return {"phi": st["phi"], "field": st["field"]}


def work(case):
    """Bytes: positions and layers (where they are new), charges in, potentials
    and fields out.  Operations of the method with boxes of 20 charges: moments
    and local expansions at every charge, the 27 neighbouring boxes' pairs, and
    per box 189 translations of 3 (p+1)^3 multiply-adds (rotated to the axis and
    back, the fewest known for exact translations)."""
    n, p1 = sum(_sizes(case)), case["p"] + 1
    new = 28 if case["call"] == "step" else 0
    out = 8 if case["call"] == "product" else 32
    each = 4 if case["form"] == "f32" and case["call"] != "product" else 8
    nbytes = n * new + n * case["nrhs"] * (8 + out * each // 8)
    flops = n * case["nrhs"] * (2 * 20 * p1 ** 2 + 27 * 20 * 20 + (8 / 7) / 20 * 189 * 6 * p1 ** 3)
    return {"bytes": nbytes, "flops": flops}


# ---- the exact potentials and fields, in 64 bits ---------------------------
# A unit charge in layer l' of three layers is seen in layer l along every path
# of reflections and transmissions between the two interfaces: images of
# amplitude prod r, t at the vertical distance h = alpha z + beta z' + gamma.

def _images(l, lp, d, eps):
    def r(i, j):
        return (eps[i] - eps[j]) / (eps[i] + eps[j])

    def t(i, j):
        return 1.0 + r(i, j)

    d0, d1 = d
    D = d0 - d1
    x = r(1, 0) * r(1, 2)
    m = 1 if x == 0.0 else min(600, int(math.ceil(math.log(1e-15) / math.log(abs(x)))) + 1)
    out = []

    def series(amp, alpha, beta, gamma):
        for n in range(m):
            out.append((amp * x ** n, alpha, beta, gamma + 2 * D * n))

    if lp == 0 and l == 0:
        out.append((r(0, 1), 1, 1, -2 * d0))
        series(t(0, 1) * r(1, 2) * t(1, 0), 1, 1, -2 * d0 + 2 * D)
    elif lp == 2 and l == 2:
        out.append((r(2, 1), -1, -1, 2 * d1))
        series(t(2, 1) * r(1, 0) * t(1, 2), -1, -1, 2 * d1 + 2 * D)
    elif lp == 0 and l == 1:
        series(t(0, 1), -1, 1, 0.0)
        series(t(0, 1) * r(1, 2), 1, 1, -2 * d1)
    elif lp == 2 and l == 1:
        series(t(2, 1), 1, -1, 0.0)
        series(t(2, 1) * r(1, 0), -1, -1, 2 * d0)
    elif lp == 0 and l == 2:
        series(t(0, 1) * t(1, 2), -1, 1, 0.0)
    elif lp == 2 and l == 0:
        series(t(2, 1) * t(1, 0), 1, -1, 0.0)
    elif lp == 1 and l == 0:
        series(t(1, 0), 1, -1, 0.0)
        series(r(1, 2) * t(1, 0), 1, 1, -2 * d1)
    elif lp == 1 and l == 2:
        series(t(1, 2), -1, 1, 0.0)
        series(r(1, 0) * t(1, 2), -1, -1, 2 * d0)
    else:
        series(r(1, 0), -1, -1, 2 * d0)
        series(r(1, 2), 1, 1, -2 * d1)
        series(x, 1, -1, 2 * D)
        series(x, -1, 1, 2 * D)
    return out


def _direct(w, q, dev):
    """Potentials [nrhs, n] and fields [nrhs, n, 3] of the charges q [nrhs, n]."""
    n = w.n
    xyz = torch.from_numpy(w.xyz).to(dev)
    layer = torch.from_numpy(w.layer).to(dev)
    phi = torch.zeros((q.shape[0], n), dtype=torch.float64, device=dev)
    fld = torch.zeros((q.shape[0], n, 3), dtype=torch.float64, device=dev)
    idx = [torch.nonzero(layer == l).ravel() for l in range(3)]
    for lp in range(3):
        s = xyz[idx[lp]]
        qs = q[:, idx[lp]].T.contiguous()
        ns = s.shape[0]
        if ns == 0:
            continue
        for l in range(3):
            imgs = _images(l, lp, [float(v) for v in w.d], [float(v) for v in w.eps])
            step = max(1, (1 << 22) // ns)
            for c in range(0, idx[l].numel(), step):
                at = idx[l][c:c + step]
                t = xyz[at]
                dx = t[:, None, 0] - s[None, :, 0]
                dy = t[:, None, 1] - s[None, :, 1]
                rho2 = dx * dx + dy * dy
                K, S, Z = (torch.zeros_like(rho2) for _ in range(3))
                if l == lp:
                    h = t[:, None, 2] - s[None, :, 2]
                    inv = torch.addcmul(rho2, h, h).rsqrt_()
                    inv[at[:, None] == idx[lp][None, :]] = 0.0
                    K += inv
                    S += inv ** 3
                    Z += inv ** 3 * h
                for amp, alpha, beta, gamma in imgs:
                    h = (alpha * t[:, 2] + gamma)[:, None] + (beta * s[:, 2])[None, :]
                    inv = torch.addcmul(rho2, h, h).rsqrt_()
                    K.add_(inv, alpha=amp)
                    inv3 = inv * inv * inv
                    S.add_(inv3, alpha=amp)
                    Z.addcmul_(inv3, h, value=amp * alpha)
                phi[:, at] += (K @ qs).T
                fld[:, at, 0] += ((S * dx) @ qs).T
                fld[:, at, 1] += ((S * dy) @ qs).T
                fld[:, at, 2] += (Z @ qs).T
    return phi / (4 * math.pi), fld / (4 * math.pi)


def exact(case, seed):
    if case["points"] == "four":
        return None  # no closed form
    pairs = sum(n * n for n in _sizes(case)) * (15.0 if case["medium"] == "contrast" else 1.0)
    if pairs > 4.5e9 or case["nrhs"] * pairs > 1e11:
        return None  # minutes of direct summation
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    phis, flds = [], []
    for w in _problems(case, seed):
        q = torch.from_numpy(w.q).to(dev) if case["nrhs"] == 1 else _charges(case, w, seed)
        phi, fld = _direct(w, q.reshape(-1, w.n), dev)
        phis.append(phi.reshape(q.shape))
        flds.append(fld.reshape(tuple(q.shape) + (3,)))
    if case["call"] == "product":
        return {"phi": phis[0].cpu().numpy()}
    if case["call"] == "batch":
        return {"phi": torch.cat(phis), "field": torch.cat([f.ravel() for f in flds])}
    return {"phi": phis[0], "field": flds[0]}
