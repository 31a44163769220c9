"""Performance cases of the lattice library: what its users have it do, through
the public entry points, from the smallest lattices to the largest.

A case is a dict of plain values with a "kind":

  operator     one application of the operator to internal fields (lqcd_dslash)
  canonical    the FP64 operator on canonical spinors: pack, apply, unpack
  setup        a new gauge field: load the links, build and invert the clover term
  sap          one Schwarz preconditioner application
  net_forward  the parallel-transport network on a batch of spinors
  net_train    one training step of that network: loss, gradients, new weights
  solve        a whole solve to a true residual of 1e-10
  batch        lattices of uneven size solved together

Links are exp(i eps H) with H random traceless Hermitian (SU(3) to FP64
accuracy), sources are complex Gaussian: the fields of this repository's
configurations and benchmark.  A solve's right-hand side is b = M x* for a
Gaussian x*, so that its solution is known.  The 64-bit reference below is
plain torch on canonical arrays (full gamma matrices, rolled lattices).
"""
import math

import torch

from paper_1103_1363_gb300 import learned, lqcd

DEV = "cuda"
C128 = torch.complex128
OPS = {"hop": lqcd.OP_HOP, "schur": lqcd.OP_SCHUR, "full": lqcd.OP_FULL}
RELIABLE = dict(reliable_interval=100, reliable_delta=0.1, check_interval=10)


def listed():
    return [
        # the operator of one small lattice of a batch: latency and launches count
        dict(name="schur_f32_8x8x8x8", kind="operator", op="schur", prec="f32", dims="8x8x8x8", nrhs=1, recon=12,
             dag=False, kappa=0.12, csw=1.0, eps=0.5),
        # the hopping term at the benchmark's size, FP32: the bandwidth figure
        dict(name="hop_f32_32x32x32x64", kind="operator", op="hop", prec="f32", dims="32x32x32x64", nrhs=1, recon=12,
             dag=False, kappa=0.1355, csw=0.0, eps=0.4),
        # 12 spin-colour sources at once in the precision of the mixed solves
        dict(name="schur_f16spinors_24x48_12rhs", kind="operator", op="schur", prec="f16spinors",
             dims="24x24x24x48", nrhs=12, recon=12, dag=True, kappa=0.135, csw=1.0, eps=0.5),
        # all operands in 16 bits on an uneven lattice (sites per parity not a multiple of a block)
        dict(name="full_f16_12x10x14x18", kind="operator", op="full", prec="f16", dims="12x10x14x18", nrhs=3,
             recon=12, dag=False, kappa=0.13, csw=1.0, eps=0.5),
        # right-hand sides of training pairs: canonical FP64 spinors through M
        dict(name="canonical_f64_16x16x16x16", kind="canonical", dims="16x16x16x16", nrhs=16, kappa=0.134, csw=1.0,
             eps=0.5),
        # a new gauge field on the even-odd configuration's lattice
        dict(name="setup_16x16x16x32", kind="setup", dims="16x16x16x32", recon=12, half=False, kappa=0.135, csw=1.0,
             eps=0.5),
        # the Schwarz preconditioner with the paper's 4^4 blocks
        dict(name="sap_16x16x16x32", kind="sap", dims="16x16x16x32", block="4x4x4x4", ncycle=5, nmr=4, recon=12,
             kappa=0.134, csw=1.0, eps=0.5),
        # the learned preconditioner as a solver applies it: one residual at a time
        dict(name="net_forward_16x16x16x16", kind="net_forward", dims="16x16x16x16", batch=1, channels="1-12-12-1",
             bf16=True, eps=0.5),
        # one step of its training
        dict(name="net_train_16x16x16x16_b16", kind="net_train", dims="16x16x16x16", batch=16, channels="1-12-12-1",
             bf16=True, eps=0.5),
        # the mixed-precision solve of the benchmark
        dict(name="solve_f16spinors_32x32x32x64", kind="solve", solver="cg_eo", inner="f16spinors",
             dims="32x32x32x64", nrhs=1, graph=False, kappa=0.1355, csw=1.0, eps=0.4),
        # three lattices of uneven size in one graph-replayed solve
        dict(name="batch_f32_uneven", kind="batch", dims="8x8x8x8,12x12x12x12,16x16x16x32",
             kappas="0.12,0.1275,0.135", inner="f32", graph=True, csw=1.0, eps=0.5),
        # flexible GCR with the Schwarz preconditioner
        dict(name="fgcr_sap_16x16x16x16", kind="solve", solver="fgcr_sap", inner="f32", dims="16x16x16x16", nrhs=1,
             graph=False, kappa=0.134, csw=1.0, eps=0.5),
    ]


def draw(rng):
    kind = rng.choices(["operator", "canonical", "setup", "sap", "net_forward", "net_train", "solve", "batch"],
                       [34, 7, 10, 10, 10, 7, 16, 6])[0]
    eps, csw = rng.choice([0.4, 0.5]), rng.choice([1.0, 1.0, 0.0])
    kappa = round(rng.uniform(0.118, 0.134), 4)
    recon = rng.choice([12, 12, 18])
    if kind == "operator":
        dims = _draw_dims(rng, 256, 2 << 20)
        most = max(1, (8 << 20) // math.prod(dims))
        prec = rng.choice([p for p in lqcd.PREC])
        if prec == "f64":
            most = min(most, 4)
        nrhs = min(rng.choice([1, 1, 1, 2, 3, 4, 5, 8, 12]), most)
        return dict(kind=kind, op=rng.choice(["hop", "schur", "schur", "full"]), prec=prec, dims=_text(dims),
                    nrhs=nrhs, recon=recon, dag=rng.random() < 0.5, kappa=kappa, csw=csw, eps=eps)
    if kind == "canonical":
        dims = _draw_dims(rng, 256, 1 << 17)
        nrhs = min(rng.choice([1, 2, 5, 16, 64]), max(1, (1 << 21) // math.prod(dims)))
        return dict(kind=kind, dims=_text(dims), nrhs=nrhs, kappa=kappa, csw=csw, eps=eps)
    if kind == "setup":
        return dict(kind=kind, dims=_text(_draw_dims(rng, 256, 1 << 19)), recon=recon, half=rng.random() < 0.5,
                    kappa=kappa, csw=1.0, eps=eps)
    if kind == "sap":
        block = rng.choice([(4, 4, 4, 4), (4, 4, 4, 4), (8, 4, 4, 4), (2, 4, 4, 2), (8, 4, 8, 4), (4, 4, 2, 6)])
        dims = [b * rng.choice([2, 2, 4]) for b in block]
        return dict(kind=kind, dims=_text(dims), block=_text(block), ncycle=rng.choice([1, 2, 4, 5]),
                    nmr=rng.choice([2, 3, 4, 5]), recon=recon, kappa=kappa, csw=csw, eps=eps)
    if kind in ("net_forward", "net_train"):
        dims = _draw_dims(rng, 256, 1 << 16)
        batch = min(rng.choice([1, 2, 3, 4, 8, 16]), max(1, (1 << 20) // math.prod(dims)))
        channels = rng.choice(["1-12-12-1", "1-12-12-1", "1-12-12-1", "1-8-8-1", "1-4-6-1"])
        return dict(kind=kind, dims=_text(dims), batch=batch, channels=channels, bf16=rng.random() < 0.8, eps=eps)
    if kind == "solve":
        solver = rng.choice(["cg_eo", "cg_eo", "cg_eo", "cg_full", "fgcr", "fgcr_sap"])
        if solver == "fgcr_sap":
            dims = [4 * rng.choice([2, 2, 4]) for _ in range(4)]
        else:
            dims = _draw_dims(rng, 256, 1 << 17)
        one = solver.startswith("fgcr")
        inner = "f32" if one else rng.choice(["f32", "f16spinors", "f16spinors", "bf16spinors", "f64"])
        nrhs = 1 if one else min(rng.choice([1, 1, 2, 4, 12]), max(1, (1 << 19) // math.prod(dims)))
        if inner == "f64":
            nrhs = min(nrhs, 2)
        return dict(kind=kind, solver=solver, inner=inner, dims=_text(dims), nrhs=nrhs,
                    graph=rng.random() < 0.6 and not one, kappa=round(rng.uniform(0.116, 0.13), 4), csw=csw, eps=0.5)
    n = rng.choice([2, 3, 4])
    return dict(kind="batch", dims=",".join(_text(_draw_dims(rng, 256, 1 << 16)) for _ in range(n)),
                kappas=",".join("%.4f" % rng.uniform(0.116, 0.13) for _ in range(n)),
                inner=rng.choice(["f32", "f16spinors"]), graph=rng.random() < 0.7, csw=1.0, eps=0.5)


def _draw_dims(rng, low, high):
    """Even extents, volumes spread over their logarithm."""
    while True:
        side = math.exp(rng.uniform(math.log(low), math.log(high)) / 4)
        dims = [max(4, 2 * round(side * rng.uniform(0.65, 1.5) / 2)) for _ in range(3)]
        dims.append(max(4, 2 * round(side * rng.uniform(0.8, 2.4) / 2)))
        if low <= math.prod(dims) <= high:
            return dims


def _text(dims):
    return "x".join(str(d) for d in dims)


def _dims(text):
    return tuple(int(d) for d in text.split("x"))


# ------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _mm(a, b):
    """Products of 3x3 matrices."""
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _dag(a):
    return a.mH


def _gauge(dims, eps, gen):
    """exp(i eps H) per link: (Lt, Lz, Ly, Lx, 4, 3, 3)."""
    lx, ly, lz, lt = dims
    h = torch.randn((lt, lz, ly, lx, 4, 8), dtype=torch.float64, device=DEV, generator=gen) * 0.5 * eps
    m = torch.zeros((lt, lz, ly, lx, 4, 3, 3), dtype=C128, device=DEV)
    s = h[..., 7] / math.sqrt(3.0)
    m[..., 0, 0], m[..., 1, 1], m[..., 2, 2] = 1j * (h[..., 2] + s), 1j * (s - h[..., 2]), -2j * s
    for (r, c), (x, y) in (((0, 1), (0, 1)), ((0, 2), (3, 4)), ((1, 2), (5, 6))):
        m[..., r, c] = torch.complex(h[..., y], h[..., x])
        m[..., c, r] = torch.complex(-h[..., y], h[..., x])
    m /= 16.0
    out = torch.eye(3, dtype=C128, device=DEV).expand_as(m).clone()
    for k in range(12, 0, -1):  # Taylor series of exp(m), then four squarings
        out = _mm(m, out) / k
        for d in range(3):
            out[..., d, d] += 1.0
    for _ in range(4):
        out = _mm(out, out)
    return out


def _spinor(dims, gen, nrhs=1, dtype=C128):
    lx, ly, lz, lt = dims
    return torch.randn((nrhs, lt, lz, ly, lx, 4, 3), dtype=dtype, device=DEV, generator=gen)


def _lattice(case, dims, links, precisions, kappa, stream=None, **kw):
    lat = lqcd.Lattice(dims, precisions=precisions, recon=case.get("recon", 12), device=DEV, stream=stream, **kw)
    lat.gauge_load(links)
    if kappa is not None:
        lat.clover_compute(kappa, case["csw"])
    lat.sync()
    return lat


def _precisions(prec):
    return ("f64",) if prec == "f64" else ("f64", "f32", prec)


def _view(lat, field, prec, nrhs, full):
    """The written values of internal fields, without the padding of the site index."""
    vh = lat.volume // 2
    stride = (vh + 127) // 128 * 128
    f = field.view(nrhs * (2 if full else 1), -1)
    if prec == "f64":
        return f.view(torch.float64).view(-1, 12, stride, 2)[:, :, :vh]
    if prec in ("f32", "f16links", "bf16links"):
        return f.view(torch.float32).view(-1, 6, stride, 4)[:, :, :vh]
    q = f[:, :48 * stride].view(torch.bfloat16 if prec.startswith("bf16") else torch.float16)
    n = f[:, 48 * stride:].view(torch.float32)
    return {"q": q.unflatten(1, (3, stride, 8))[:, :, :vh], "norm": n[:, :vh]}


def _solve_params(case):
    solver = case.get("solver", "cg_eo")
    kind = {"cg_eo": lqcd.SOLVER_CG_EO, "cg_full": lqcd.SOLVER_CG_FULL}.get(solver, lqcd.SOLVER_FGCR)
    p = dict(solver=kind, inner_prec=case["inner"], use_graph=int(case["graph"]), maxiter=20000)
    if kind == lqcd.SOLVER_FGCR:
        p["nkrylov"] = 20
    else:
        p.update(RELIABLE)
    return p


def _weights(channels, gen):
    """Complex Gaussian weights plus the spin identity on hop 0 of channel 0."""
    parts = []
    for cin, cout in zip(channels, channels[1:]):
        w = 0.02 * torch.view_as_complex(torch.randn((9, 4 * cout, 4 * cin, 2), device=DEV, generator=gen))
        w[0, :4, :4] += torch.eye(4, device=DEV)
        parts.append(w.reshape(-1))
    return torch.cat(parts)


def _net(case, seed):
    gen = _gen(seed)
    dims = _dims(case["dims"])
    links = _gauge(dims, case["eps"], gen)
    lat = _lattice(case, dims, links, ("f64", "f32"), None)
    channels = tuple(int(c) for c in case["channels"].split("-"))
    net = lqcd.Net(lat, channels, bf16=case["bf16"], max_batch=case["batch"])
    net.set_weights(_weights(channels, gen))
    r = _spinor(dims, gen, case["batch"], torch.complex64)
    return lat, net, r, gen


def prepare(case, seed):
    kind, gen = case["kind"], _gen(seed)
    s = dict(case=case, kind=kind)
    if kind == "operator":
        dims, prec, nrhs = _dims(case["dims"]), case["prec"], case["nrhs"]
        links = _gauge(dims, case["eps"], gen)
        lat = _lattice(case, dims, links, _precisions(prec), case["kappa"], max_nrhs=nrhs)
        del links
        full = case["op"] == "full"
        src = _spinor(dims, gen, nrhs)
        fin, fout = lat.new_field(prec, nrhs, full), lat.new_field(prec, nrhs, full)
        parity = 0 if case["op"] == "hop" else 1
        lat.pack(fin, src, -1 if full else 1, prec, nrhs)
        s.update(lat=lat, fin=fin, fout=fout, parity=parity, out=_view(lat, fout, prec, nrhs, full),
                 csw=case["csw"], kappa=case["kappa"])
    elif kind == "canonical":
        dims = _dims(case["dims"])
        links = _gauge(dims, case["eps"], gen)
        lat = _lattice(case, dims, links, ("f64",), case["kappa"], max_nrhs=case["nrhs"])
        src = _spinor(dims, gen, case["nrhs"])
        s.update(lat=lat, src=src, out=torch.empty_like(src))
    elif kind == "setup":
        dims = _dims(case["dims"])
        links = _gauge(dims, case["eps"], gen)
        precs = ("f64", "f32", "f16") if case["half"] else ("f64", "f32")
        lat = lqcd.Lattice(dims, precisions=precs, recon=case["recon"], device=DEV)
        src = _spinor(dims, gen)
        fin = {p: lat.new_field(p) for p in ("f64", "f32")}
        fout = {k: lat.new_field(k[1]) for k in (("a", "f64"), ("ainv", "f64"), ("ainv", "f32"), ("hop", "f32"))}
        s.update(lat=lat, links=links, src=src, fin=fin, fout=fout,
                 out={"%s_%s" % k: _view(lat, v, k[1], 1, False) for k, v in fout.items()})
    elif kind == "sap":
        dims = _dims(case["dims"])
        links = _gauge(dims, case["eps"], gen)
        lat = _lattice(case, dims, links, ("f64", "f32"), case["kappa"])
        r, z = lat.new_field("f32", full=True), lat.new_field("f32", full=True)
        lat.pack(r, _spinor(dims, gen), -1, "f32")
        s.update(lat=lat, r=r, z=z, out=_view(lat, z, "f32", 1, True))
    elif kind in ("net_forward", "net_train"):
        lat, net, r, gen = _net(case, seed)
        s.update(lat=lat, net=net, r=r)
        if kind == "net_forward":
            s["out"] = torch.empty_like(r)
        else:
            s["e"] = _spinor(_dims(case["dims"]), gen, case["batch"], torch.complex64)
    elif kind == "solve":
        dims = _dims(case["dims"])
        links = _gauge(dims, case["eps"], gen)
        stream = torch.cuda.Stream(device=DEV)
        torch.cuda.synchronize()
        fgcr = case["solver"].startswith("fgcr")
        precs = _precisions(case["inner"])
        lat = _lattice(case, dims, links, precs, case["kappa"], stream=stream, max_nrhs=case["nrhs"],
                       gcr_nkrylov=20 if fgcr else 0)
        if case["solver"] == "fgcr_sap":
            lat.set_sap((4, 4, 4, 4), 5, 4)
        b = _matrix(links, _clover(links, case["kappa"], case["csw"]), case["kappa"], _spinor(dims, gen, case["nrhs"]))
        s.update(lat=lat, b=b, x=torch.zeros_like(b), params=_solve_params(case))
    else:
        stream = torch.cuda.Stream(device=DEV)
        lats, bs = [], []
        for dims, kappa in zip(case["dims"].split(","), case["kappas"].split(",")):
            dims, kappa = _dims(dims), float(kappa)
            links = _gauge(dims, case["eps"], gen)
            torch.cuda.synchronize()
            lats.append(_lattice(case, dims, links, _precisions(case["inner"]), kappa, stream=stream))
            bs.append(_matrix(links, _clover(links, kappa, case["csw"]), kappa, _spinor(dims, gen)))
        s.update(lats=lats, bs=bs, xs=[torch.zeros_like(b) for b in bs], tols=[1e-10] * len(bs),
                 params=lqcd.solver_params(**_solve_params(case)))
    torch.cuda.synchronize()
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "operator":
        s["lat"].dslash(s["fout"], s["fin"], s["parity"], s["kappa"], s["csw"], OPS[case["op"]], case["dag"],
                        case["prec"], case["nrhs"])
        return s["out"]
    if kind == "canonical":
        learned.apply_full_operator(s["lat"], s["out"], s["src"], case["nrhs"])
        return s["out"]
    if kind == "setup":
        lat, fin, fout = s["lat"], s["fin"], s["fout"]
        lat.gauge_load(s["links"])
        lat.clover_compute(case["kappa"], case["csw"])
        for p in ("f64", "f32"):
            lat.pack(fin[p], s["src"], 1, p)
        lat.clover_apply(fout["a", "f64"], fin["f64"], 1, 0, "f64")
        lat.clover_apply(fout["ainv", "f64"], fin["f64"], 1, 1, "f64")
        lat.clover_apply(fout["ainv", "f32"], fin["f32"], 1, 1, "f32")
        lat.dslash(fout["hop", "f32"], fin["f32"], 0, prec="f32")
        return s["out"]
    if kind == "sap":
        s["lat"].sap_apply(s["z"], s["r"], _dims(case["block"]), case["ncycle"], case["nmr"])
        return s["out"]
    if kind == "net_forward":
        s["net"].forward(s["out"], s["r"], case["batch"])
        return s["out"]
    if kind == "net_train":
        # the small step of the end of a learning-rate schedule: weights hardly move between passes
        loss = s["net"].train_step(s["r"], s["e"], case["batch"], lr=1e-6)
        weights, grad = s["net"].get_weights(grad=True)
        return {"loss": loss, "grad": grad, "weights": weights}
    if kind == "solve":
        s["lat"].solve(s["x"], s["b"], 1e-10, case["nrhs"], **s["params"])
        return s["x"]
    lqcd.lqcd_solve_batch([lat.ctx for lat in s["lats"]], s["xs"], s["bs"], s["tols"], s["params"])
    return s["xs"]


# ------------------------------------------------------------- work

_SPINOR = {"f64": 192, "f32": 96, "f16links": 96, "bf16links": 96}
_LINK = {"f64": 144, "f32": 48, "f16spinors": 48, "bf16spinors": 48}


def _site_bytes(prec, recon):
    """Bytes per site of a spinor, a link and a clover entry in a precision mode."""
    spinor, link = _SPINOR.get(prec, 52), _LINK.get(prec, 24)
    return spinor, link if prec == "f64" or recon == 12 else link * 3 // 2, {144: 576, 48: 288, 24: 144}[link]


def _cg_iterations(volume):
    """Iterations of a mixed solve to 1e-10 that these sizes take at least (it grows slowly with the lattice)."""
    return 50 if volume <= 1 << 12 else 70 if volume <= 1 << 15 else 100 if volume <= 1 << 18 else 300


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [work(dict(case, kind="solve", solver="cg_eo", dims=d, nrhs=1)) for d in case["dims"].split(",")]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    dims = _dims(case["dims"])
    v = math.prod(dims)
    vh = v // 2
    if kind == "operator":
        n = case["nrhs"]
        spinor, link, clover = _site_bytes(case["prec"], case["recon"])
        clover = clover if case["csw"] and case["op"] != "hop" else 0
        if case["op"] == "hop":
            return {"bytes": vh * (8 * link + 2 * n * spinor), "flops": vh * n * 1320}
        if case["op"] == "schur":  # links of both parities and A_ee^-1, A_oo once; odd field in and out
            return {"bytes": vh * (8 * link + 2 * clover + 2 * n * spinor),
                    "flops": vh * n * (2 * 1320 + (1008 if clover else 0) + 48)}
        return {"bytes": v * (4 * link + clover + 2 * n * spinor),
                "flops": v * n * (1320 + (504 if clover else 0) + 48)}
    if kind == "canonical":
        return {"bytes": v * (2 * case["nrhs"] * 192 + 576 + (576 if case["csw"] else 0)),
                "flops": v * case["nrhs"] * 1872}
    if kind == "setup":
        # links in, the FP64 and FP32 links and clover blocks (A and its inverse) out
        low = 4 * (48 if case["recon"] == 12 else 72) + 2 * 288
        return {"bytes": v * (576 + 576 + 2 * 576 + low + (low // 2 if case["half"] else 0)), "flops": v * 20000}
    if kind == "sap":
        # each cycle updates every site once: residual, correction and links in, residual and correction out
        link = 48 if case["recon"] == 12 else 72
        once = 4 * link + (288 if case["csw"] else 0) + 4 * 96
        step = 13 * 66 + (504 if case["csw"] else 0) + 384
        return {"bytes": v * (once * case["ncycle"] + 2 * 96),
                "flops": v * case["ncycle"] * case["nmr"] * step}
    if kind in ("net_forward", "net_train"):
        ch = [int(c) for c in case["channels"].split("-")]
        b = case["batch"]
        macs = sum(9 * 16 * i * o for i, o in zip(ch, ch[1:]))
        flops = v * b * (8 * 3 * macs + sum(8 * 4 * i * 66 for i in ch[:-1]))
        nbytes = v * (2 * b * 96 + 192)
        return {"bytes": nbytes * (1 if kind == "net_forward" else 3),
                "flops": flops * (1 if kind == "net_forward" else 3)}
    spinor, link, clover = _site_bytes(case["inner"], 12)
    clover = clover if case["csw"] else 0
    n, its = case["nrhs"], _cg_iterations(v)
    if case["solver"].startswith("fgcr"):
        its = 11 if case["solver"] == "fgcr_sap" else its
        return {"bytes": v * its * (4 * 48 + clover + 4 * 96), "flops": v * its * (1320 + 504)}
    # one iteration: four sweeps over the links and the clover term, the vectors p, r, x
    per = 4 * (8 * link + clover) + n * (8 * spinor + 4 * (192 if case["inner"] == "f64" else 96))
    per = per if case["solver"] == "cg_eo" else 2 * per
    return {"bytes": vh * per * its, "flops": vh * its * n * 4 * 1320 * (1 if case["solver"] == "cg_eo" else 2)}


# ------------------------------------------------------------- 64-bit reference

_I = 1j
_GAMMA = [  # DeGrand-Rossi basis: nonzero entry of each row as (column, value)
    [(3, _I), (2, _I), (1, -_I), (0, -_I)],
    [(3, -1), (2, 1), (1, 1), (0, -1)],
    [(2, _I), (3, -_I), (0, -_I), (1, _I)],
    [(2, 1), (3, 1), (0, 1), (1, 1)],
]


def _gamma(mu):
    g = torch.zeros((4, 4), dtype=C128, device=DEV)
    for r, (c, v) in enumerate(_GAMMA[mu]):
        g[r, c] = v
    return g


def _axis(mu):
    return -3 - mu  # of a spinor (..., Lt, Lz, Ly, Lx, 4, 3)


def _cross(psi, mu, index):
    """The antiperiodic sign of hops across the t boundary."""
    if mu == 3:
        psi.select(_axis(3), index).neg_()
    return psi


def _colour(u, psi):
    return sum(u[..., None, :, b] * psi[..., :, b, None] for b in range(3))


def _forward(links, psi, mu):
    """U_mu(x) psi(x + mu)."""
    return _colour(links[..., mu, :, :], _cross(torch.roll(psi, -1, _axis(mu)), mu, -1))


def _backward(links, psi, mu):
    """U_mu(x - mu)^dag psi(x - mu)."""
    return _cross(torch.roll(_colour(_dag(links[..., mu, :, :]), psi), 1, _axis(mu)), mu, 0)


def _spin(mu, psi):
    rows = [v * psi[..., c, :] for c, v in _GAMMA[mu]]
    return torch.stack(rows, -2)


def _hop(links, psi):
    out = torch.zeros_like(psi)
    for mu in range(4):
        f, b = _forward(links, psi, mu), _backward(links, psi, mu)
        out += f
        out += b
        out += _spin(mu, b - f)
    return out


def _gamma5(psi):
    out = psi.clone()
    out[..., 2:, :] *= -1
    return out


def _clover(links, kappa, csw):
    """A as two 6x6 blocks per site, (Lt, Lz, Ly, Lx, 2, 6, 6); None for csw = 0."""
    if csw == 0:
        return None

    def shift(m, mu, d):  # m(x + d mu) on (Lt, Lz, Ly, Lx, 3, 3)
        return torch.roll(m, -d, -3 - mu)

    u = [links[..., mu, :, :] for mu in range(4)]
    a = torch.zeros(links.shape[:4] + (2, 2, 3, 2, 3), dtype=C128, device=DEV)
    for mu in range(4):
        for nu in range(mu + 1, 4):
            q = _mm(_mm(u[mu], shift(u[nu], mu, 1)), _dag(_mm(u[nu], shift(u[mu], nu, 1))))
            m_mu, m_nu = shift(u[mu], mu, -1), shift(u[nu], nu, -1)
            n_mu = shift(u[nu], mu, -1)  # U_nu(x - mu)
            u_nu = shift(u[mu], nu, -1)  # U_mu(x - nu)
            q += _mm(_mm(u[nu], _dag(shift(m_mu, nu, 1))), _mm(_dag(n_mu), m_mu))
            q += _mm(_dag(_mm(shift(n_mu, nu, -1), m_mu)), _mm(shift(m_mu, nu, -1), m_nu))
            q += _mm(_mm(_dag(m_nu), u_nu), _mm(shift(m_nu, mu, 1), _dag(u[mu])))
            f = (q - _dag(q)) / 8
            f = f - torch.eye(3, dtype=C128, device=DEV) * f.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3
            sigma = 0.5j * (_gamma(mu) @ _gamma(nu) - _gamma(nu) @ _gamma(mu))
            for blk in range(2):
                for r in range(2):
                    for c in range(2):
                        w = sigma[2 * blk + r, 2 * blk + c].item()
                        if w != 0:
                            a[..., blk, r, :, c, :] += 1j * kappa * csw * w * f
    a = a.reshape(links.shape[:4] + (2, 6, 6))
    return a + torch.eye(6, dtype=C128, device=DEV)


def _apply_clover(a, psi):
    if a is None:
        return psi.clone()
    v = psi.reshape(psi.shape[:-2] + (2, 6))
    return sum(a[..., :, k] * v[..., k, None] for k in range(6)).reshape(psi.shape)


def _matrix(links, a, kappa, psi):
    """M psi for each right-hand side."""
    return torch.stack([_apply_clover(a, p) - kappa * _hop(links, p) for p in psi])


def _parity(dims):
    lx, ly, lz, lt = dims
    t, z, y, x = torch.meshgrid(*(torch.arange(n, device=DEV) for n in (lt, lz, ly, lx)), indexing="ij")
    return (x + y + z + t) % 2


def _restrict(psi, dims, par):
    return psi * (_parity(dims) == par)[..., None, None]


def _internal(psi, dims, prec, parity):
    """Canonical spinors in the layout of _view()."""
    out = []
    for p in psi:
        for par in (0, 1) if parity < 0 else (parity,):
            out.append(torch.view_as_real(p.reshape(-1, 12)[(_parity(dims) == par).reshape(-1)]).reshape(-1, 24))
    v = torch.stack(out)

    def chunks(w, k):
        return w.unflatten(2, (24 // k, k)).transpose(1, 2)

    if prec == "f64":
        return chunks(v, 2)
    if prec in ("f32", "f16links", "bf16links"):
        return chunks(v, 4)
    n = v.abs().amax(2)
    return {"q": chunks(v / n[..., None], 8), "norm": n}


def _sap(links, a, kappa, r, dims, block, ncycle, nmr):
    lx, ly, lz, lt = dims
    grids = torch.meshgrid(*(torch.arange(n, device=DEV) for n in (lt, lz, ly, lx)), indexing="ij")
    coords = grids[::-1]  # x, y, z, t
    colour = sum(c // b for c, b in zip(coords, block)) % 2
    number = torch.zeros_like(colour)
    for c, b, n in zip(coords, block, dims):
        number = number * (n // b) + c // b
    first = [(c % b == 0)[..., None, None] for c, b in zip(coords, block)]
    last = [(c % b == b - 1)[..., None, None] for c, b in zip(coords, block)]
    number = number.reshape(-1)
    blocks = int(number.max()) + 1

    def dot(u, v):  # per block, spread over its sites
        d = (u.conj() * v).reshape(number.numel(), 12).sum(1)
        return torch.zeros(blocks, dtype=C128, device=DEV).index_add_(0, number, d)[number].reshape(lt, lz, ly, lx)[..., None, None]

    def inside(v):  # the operator without the hops that leave a block
        h = torch.zeros_like(v)
        for mu in range(4):
            f = torch.where(last[mu], 0, _forward(links, v, mu))
            b = torch.where(first[mu], 0, _backward(links, v, mu))
            h += f + b + _spin(mu, b - f)
        return _apply_clover(a, v) - kappa * h

    z = torch.zeros_like(r)
    for _ in range(ncycle):
        for par in range(2):
            here = (colour == par)[..., None, None]
            rho = torch.where(here, r - (_apply_clover(a, z) - kappa * _hop(links, z)), 0)
            delta = torch.zeros_like(rho)
            for _ in range(nmr):
                q = inside(rho)
                alpha = torch.where(here, dot(q, rho) / torch.where(here, dot(q, q), 1), 0)
                delta = delta + alpha * rho
                rho = rho - alpha * q
            z = z + delta
    return z


def _network(links, weights, channels, psi):
    """One item: (Lt, Lz, Ly, Lx, 4, 3) -> the same."""
    act, at = psi, 0
    lattice = psi.shape[:4]
    for cin, cout in zip(channels, channels[1:]):
        w = weights[at:at + 9 * 16 * cin * cout].reshape(9, 4 * cout, 4 * cin)
        at += 9 * 16 * cin * cout
        v = act.reshape(lattice + (4 * cin, 3))
        out = torch.matmul(w[0], v)
        for mu in range(4):
            out = out + torch.matmul(w[2 * mu + 1], _forward(links, v, mu))
            out = out + torch.matmul(w[2 * mu + 2], _backward(links, v, mu))
        act = out
    return act.reshape(lattice + (4, 3))


def exact(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind == "solve":
        dims = _dims(case["dims"])
        _gauge(dims, case["eps"], gen)
        return _spinor(dims, gen, case["nrhs"])
    if kind == "batch":
        out = []
        for dims in case["dims"].split(","):
            _gauge(_dims(dims), case["eps"], gen)
            out.append(_spinor(_dims(dims), gen))
        return out
    dims = _dims(case["dims"])
    links = _gauge(dims, case["eps"], gen)
    if kind == "operator":
        kappa, prec = case["kappa"], case["prec"]
        a = _clover(links, kappa, case["csw"]) if case["op"] != "hop" else None
        ainv = torch.linalg.inv(a) if a is not None and case["op"] == "schur" else None
        out = []
        for psi in _spinor(dims, gen, case["nrhs"]):
            psi = _gamma5(psi) if case["dag"] else psi
            if case["op"] == "hop":
                v = _hop(links, _restrict(psi, dims, 1))
            elif case["op"] == "schur":
                psi = _restrict(psi, dims, 1)
                v = _apply_clover(a, psi) - kappa * kappa * _hop(links, _apply_clover(ainv, _hop(links, psi)))
            else:
                v = _apply_clover(a, psi) - kappa * _hop(links, psi)
            out.append(_gamma5(v) if case["dag"] else v)
        return _internal(out, dims, prec, {"hop": 0, "schur": 1, "full": -1}[case["op"]])
    if kind == "canonical":
        return _matrix(links, _clover(links, case["kappa"], case["csw"]), case["kappa"], _spinor(dims, gen, case["nrhs"]))
    if kind == "setup":
        psi = _spinor(dims, gen)[0]
        a = _clover(links, case["kappa"], case["csw"])
        ax, ainvx = _apply_clover(a, psi), _apply_clover(torch.linalg.inv(a), psi)
        return {"a_f64": _internal([ax], dims, "f64", 1), "ainv_f64": _internal([ainvx], dims, "f64", 1),
                "ainv_f32": _internal([ainvx], dims, "f32", 1),
                "hop_f32": _internal([_hop(links, _restrict(psi, dims, 1))], dims, "f32", 0)}
    if kind == "sap":
        a = _clover(links, case["kappa"], case["csw"])
        z = _sap(links, a, case["kappa"], _spinor(dims, gen)[0], dims, _dims(case["block"]), case["ncycle"], case["nmr"])
        return _internal([z], dims, "f32", -1)
    channels = tuple(int(c) for c in case["channels"].split("-"))
    weights = _weights(channels, gen).to(C128)
    r = _spinor(dims, gen, case["batch"], torch.complex64).to(C128)
    if kind == "net_forward":
        return torch.stack([_network(links, weights, channels, p) for p in r])
    e = _spinor(dims, gen, case["batch"], torch.complex64).to(C128)
    weights.requires_grad_(True)
    loss = 0.0
    for p, t in zip(r, e):
        part = (_network(links, weights, channels, p) - t).abs().square().sum() / t.abs().square().sum() / case["batch"]
        part.backward()
        loss += part.item()
    return {"loss": loss, "grad": weights.grad, "weights": None}
