"""The work that a program built on this solver has it do, as cases that can be timed and compared.

A case is a dict of plain values; `prepare` makes what the program holds before the call (an
assembled scatterer, a batch, blocks in device memory), `run` is one pass through the public entry
points, and `work` what that pass cannot do without.  Five kinds:

  assemble    a new scatterer: create, assemble on the device, first steps of its march
  march       a new batch of incident waves on an assembled scatterer (every path: FP64, FP32, the
              64-wave tensor-core paths; dense or factored history; direct or GMRES solve), with
              the far field of the currents where directions are asked for
  batch       several uneven scatterers advanced together
  block_gemv  the stand-alone history sum on blocks that the caller holds
  mlp_train   training of the learned GMRES guess

A scatterer is assembled once per process and kept: a user marches many excitations on it, and the
seed of a march draws the excitation.  The time of the assembly itself is what `assemble` measures.
"""
import math

import numpy as np
import torch

from paper_2312_06367_gb300 import Batch, Solver, block_gemv, mlp_train

DEV = "cuda"


# ---------------------------------------------------------------- meshes
def _subdivide(V, F, project):
    V, mid, out = [tuple(v) for v in V], {}, []

    def midpoint(a, b):
        key = (min(a, b), max(a, b))
        if key not in mid:
            p = [(x + y) / 2 for x, y in zip(V[a], V[b])]
            r = math.sqrt(sum(x * x for x in p)) if project else 1.0
            mid[key] = len(V)
            V.append(tuple(x / r for x in p))
        return mid[key]

    for a, b, c in F:
        ab, bc, ca = midpoint(a, b), midpoint(b, c), midpoint(c, a)
        out += [(a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca)]
    return V, out


def _outward(V, F, centre):
    V, F = np.asarray(V, dtype=np.float64), np.asarray(F, dtype=np.int32)
    a, b, c = V[F[:, 0]], V[F[:, 1]], V[F[:, 2]]
    flip = np.einsum("ij,ij->i", np.cross(b - a, c - a), (a + b + c) / 3 - centre((a + b + c) / 3)) < 0
    F[flip] = F[flip][:, [0, 2, 1]]
    return V, F


def _mesh(shape, level, nu, nv):
    """sphere: subdivided icosahedron (30 * 4^level edges); ellipsoid: subdivided octahedron with
    semi-axes (2, 1, 0.5) (12 * 4^level edges); torus: nu x nv grid, radii 1 and 0.4 (3 nu nv edges,
    most of them not a multiple of four)."""
    if shape == "torus":
        V = [((1 + 0.4 * math.cos(2 * math.pi * j / nv)) * math.cos(2 * math.pi * i / nu),
              (1 + 0.4 * math.cos(2 * math.pi * j / nv)) * math.sin(2 * math.pi * i / nu),
              0.4 * math.sin(2 * math.pi * j / nv)) for i in range(nu) for j in range(nv)]
        F = []
        for i in range(nu):
            for j in range(nv):
                a, b = i * nv + j, ((i + 1) % nu) * nv + j
                c, d = ((i + 1) % nu) * nv + (j + 1) % nv, i * nv + (j + 1) % nv
                F += [(a, b, c), (a, c, d)]

        def ring(g):
            r = g * np.array([1.0, 1.0, 0.0])
            return r / np.linalg.norm(r, axis=1, keepdims=True)
        return _outward(V, F, ring)
    if shape == "ellipsoid":
        V = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        F = [(x, y, z) for x in (0, 1) for y in (2, 3) for z in (4, 5)]
    else:
        t = (1 + math.sqrt(5)) / 2
        V = [p for a in (-1, 1) for b in (-t, t) for p in ((a, b, 0), (0, a, b), (b, 0, a))]
        V = [tuple(x / math.sqrt(1 + t * t) for x in p) for p in V]
        d = [[sum((x - y) ** 2 for x, y in zip(p, q)) for q in V] for p in V]
        e2 = min(x for r in d for x in r if x > 1e-9) * 1.01
        F = [(i, j, k) for i in range(12) for j in range(i) for k in range(j) if max(d[i][j], d[j][k], d[i][k]) < e2]
    for _ in range(level):
        V, F = _subdivide(V, F, True)
    V, F = _outward(V, F, lambda g: 0.0)
    return (V * np.array([2.0, 1.0, 0.5]) if shape == "ellipsoid" else V), F


def _sizes(m):
    """(edges, triangles, lags K) of a scatterer."""
    if m["shape"] == "torus":
        ne, diam = 3 * m["nu"] * m["nv"], 2.8
    else:
        ne, diam = (30 if m["shape"] == "sphere" else 12) * 4 ** m["level"], 2.0 if m["shape"] == "sphere" else 4.0
    return ne, 2 * ne // 3, math.ceil(diam / m["dt"] + 2)


def _waves(R, seed):
    """R plane waves of random directions and polarisations; a pulse that rises within the march."""
    g = np.random.Generator(np.random.PCG64(seed))
    k = g.standard_normal((R, 3))
    k /= np.linalg.norm(k, axis=1, keepdims=True)
    p = g.standard_normal((R, 3))
    p -= np.sum(p * k, axis=1, keepdims=True) * k
    p /= np.linalg.norm(p, axis=1, keepdims=True)
    return {"k": k, "p": p, "amp": g.uniform(0.5, 1.5, R), "t0": g.uniform(3.0, 5.0, R), "sigma": g.uniform(1.2, 1.8, R)}


# ---------------------------------------------------------------- the listed cases
def _march(name, shape, prec, R, nt, dt, alpha=1.0, level=0, nu=0, nv=0, solver="direct", form="dense", ndir=0):
    return dict(name=name, kind="march", shape=shape, level=level, nu=nu, nv=nv, dt=dt, alpha=alpha, prec=prec, R=R,
                nt=nt, solver=solver, form=form, ndir=ndir)


def listed():
    return [
        # the smallest scatterer a study starts with, from its mesh to the first currents
        dict(name="assemble_sphere120_fp64", kind="assemble", shape="sphere", level=1, nu=0, nv=0, dt=0.4, alpha=1.0,
             prec="fp64", R=1, nt=20),
        # an ordinary mesh: what every change of geometry or time step costs its user
        dict(name="assemble_sphere480_fp64", kind="assemble", shape="sphere", level=2, nu=0, nv=0, dt=0.4, alpha=1.0,
             prec="fp64", R=1, nt=20),
        # one wave on a small sphere in full precision: 300 short steps, launches and latency count
        _march("march_sphere480_fp64", "sphere", "fp64", 1, 300, 0.2, level=2),
        # a long march at a large time step (four lags), single precision
        _march("march_torus864_fp32", "torus", "fp32", 1, 1000, 2.0, alpha=0.5, nu=24, nv=12),
        # a history larger than the L2 cache (43 blocks), one wave
        _march("march_sphere1920_fp32", "sphere", "fp32", 1, 200, 0.05, level=3),
        # eight waves together on the same history (training trajectories, monostatic sweeps)
        _march("march_sphere1920_fp32_r8", "sphere", "fp32", 8, 100, 0.05, level=3),
        # 64 directions on the tensor cores: the batched sweep
        _march("march_sphere1920_fp16x3_r64", "sphere", "fp16x3", 64, 100, 0.05, level=3),
        # the iterative solve with the extrapolated guess
        _march("march_ellipsoid768_gmres_fp32", "ellipsoid", "fp32", 1, 100, 0.2, level=3, solver="gmres"),
        # the factored history, then the far field of the currents over a cut of directions
        _march("scatter_sphere480_factored_fp64", "sphere", "fp64", 1, 300, 0.2, level=2, form="factored", ndir=181),
        # several uneven scatterers stepped together
        dict(name="batch_uneven5_fp32", kind="batch", members="sphere2:0.2,torus16x8:1.0,sphere1:0.4,torus10x5:1.0,ellipsoid2:0.3",
             nt=100),
        # the history sum of a large problem on blocks that the caller holds (41 lags, 7680 edges)
        dict(name="block_gemv_fp32_7680", kind="block_gemv", dtype="float32", nblk=41, n=7680, R=1),
        # one pass of training of the learned guess over a small trajectory's samples
        dict(name="mlp_train_262144", kind="mlp_train", n=262144, batch=4096, epochs=1),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _draw_scatterer(rng, tori=True):
    shape = rng.choice(["sphere", "ellipsoid", "torus"] if tori else ["sphere", "ellipsoid"])
    if shape == "torus":
        nv = rng.randint(4, 8)
        return dict(shape=shape, level=0, nu=rng.randint(nv + 2, 2 * nv), nv=nv, dt=round(rng.uniform(1.0, 3.0), 3), alpha=0.5)
    if shape == "ellipsoid":
        return dict(shape=shape, level=rng.randint(1, 2), nu=0, nv=0, dt=round(_log(rng, 0.3, 0.8), 3), alpha=1.0)
    return dict(shape=shape, level=rng.randint(1, 2), nu=0, nv=0, dt=round(_log(rng, 0.4, 0.8), 3), alpha=1.0)


def draw(rng):
    kind = rng.choice(["assemble", "assemble", "march", "march", "march", "march", "march", "batch", "block_gemv", "mlp_train"])
    if kind == "assemble":
        return dict(kind=kind, prec=rng.choice(["fp64", "fp32"]), R=rng.randint(1, 4), nt=rng.randint(10, 30), **_draw_scatterer(rng))
    if kind == "march":
        how = rng.choice(["fp64", "fp64", "fp32", "fp32", "fp16x3", "bf16x3"])
        R = 64 if how.endswith("x3") else rng.choice([1, 1, 2, 3, 5, 8])
        c = dict(kind=kind, prec=how, R=R, nt=int(_log(rng, 20, 300)), solver="direct", form="dense", ndir=0)
        c.update(_draw_scatterer(rng, tori=R != 64))
        if R != 64:
            extra = rng.choice(["", "", "gmres", "factored", "far"])
            if extra == "gmres" and _sizes(c)[2] >= 5:
                c["solver"] = "gmres"
            elif extra == "factored":
                c["form"] = "factored"
            elif extra == "far":
                c["ndir"] = rng.randint(1, 361)
        return c
    if kind == "batch":
        menu = ["sphere1:0.4", "sphere1:0.7", "ellipsoid1:0.5", "ellipsoid2:0.3", "torus10x5:1.0", "torus9x4:2.0", "torus11x6:1.5", "sphere2:0.5"]
        return dict(kind=kind, members=",".join(rng.sample(menu, rng.randint(2, 6))), nt=int(_log(rng, 20, 150)))
    if kind == "block_gemv":
        dtype, R = rng.choice(["float32", "float64"]), rng.choice([1, 1, 2, 3, 4, 6, 8])
        n = int(_log(rng, 100, 7680))
        most = 2e9 / (n * n * (4 if dtype == "float32" else 8) * R)
        return dict(kind=kind, dtype=dtype, nblk=max(1, min(rng.randint(1, 48), int(most))), n=n, R=R)
    n = int(_log(rng, 2000, 262144))
    return dict(kind=kind, n=n, batch=max(int(_log(rng, 256, 8192)), n // 64), epochs=rng.randint(1, 2))


# ---------------------------------------------------------------- state
_kept = {}      # assembled scatterers and batches of this process


def _solver(c, prec, R, role):
    key = (c["shape"], c["level"], c["nu"], c["nv"], c["dt"], c["alpha"], role)
    if key not in _kept:
        V, F = _mesh(c["shape"], c["level"], c["nu"], c["nv"])
        _kept[key] = Solver(V, F, dt=c["dt"], nt=1, alpha=c["alpha"], precision=prec, R=R).assemble()
        _kept[key].planned = (prec, R, "direct", "dense")
    return _kept[key]


def _plan(s, c):
    """Give the kept scatterer the plan of this case (nothing where it has it already)."""
    want = (c["prec"], c["R"], c["solver"], c["form"])
    if s.planned != want:
        if s.planned[2] != "direct":
            s.set_solver("direct")
        if s.planned[3] != "dense":
            s.set_history_form("dense")
        s.replan(c["prec"], c["R"])
        if c["form"] != "dense":
            s.set_history_form(c["form"])
        if c["solver"] == "gmres":
            s.set_solver("gmres", "extrap", 1e-8)
        s.planned = want


def _member(text):
    shape, dt = text.split(":")
    if shape.startswith("torus"):
        nu, nv = (int(x) for x in shape[5:].split("x"))
        return dict(shape="torus", level=0, nu=nu, nv=nv, dt=float(dt), alpha=0.5)
    return dict(shape=shape[:-1], level=int(shape[-1]), nu=0, nv=0, dt=float(dt), alpha=1.0)


def prepare(case, seed):
    c = case
    if c["kind"] == "assemble":
        V, F = _mesh(c["shape"], c["level"], c["nu"], c["nv"])
        g = np.random.Generator(np.random.PCG64(seed))
        V = V * g.uniform(0.97, 1.03, (V.shape[0], 1)) if c["shape"] != "torus" else V * g.uniform(0.97, 1.03)
        out = torch.zeros((c["nt"], c["R"], F.shape[0] * 3 // 2), device=DEV,
                          dtype=torch.float64 if c["prec"] == "fp64" else torch.float32)
        return dict(case=c, V=V, F=F, pw=_waves(c["R"], seed + 1), out=out)
    if c["kind"] == "march":
        s = _solver(c, "fp64", 1, "march")
        _plan(s, c)
        g = np.random.Generator(np.random.PCG64(seed + 2))
        rhat = g.standard_normal((max(1, c["ndir"]), 3))
        rhat /= np.linalg.norm(rhat, axis=1, keepdims=True)
        out = torch.zeros((c["nt"], c["R"], s.ne), dtype=s.dtype, device=DEV)
        return dict(case=c, s=s, pw=_waves(c["R"], seed), out=out, rhat=rhat)
    if c["kind"] == "batch":
        ms = [_member(t) for t in c["members"].split(",")]
        ss = [_solver(m, "fp32", 1, "batch") for m in ms]
        pw = [_waves(1, seed + 10 * i) for i in range(len(ss))]
        if c["members"] not in _kept:
            for s, w in zip(ss, pw):
                s.set_excitation(w)
            _kept[c["members"]] = Batch(ss)
        return dict(case=c, ss=ss, b=_kept[c["members"]], pw=pw,
                    outs=[torch.zeros((c["nt"], 1, s.ne), dtype=s.dtype, device=DEV) for s in ss])
    g = torch.Generator(device=DEV).manual_seed(seed)
    if c["kind"] == "block_gemv":
        dt, n = getattr(torch, c["dtype"]), c["n"]
        B = torch.empty((c["nblk"], n, n), dtype=dt, device=DEV).normal_(0.0, 1.0 / math.sqrt(n), generator=g)
        X = torch.empty((c["nblk"], c["R"], n), dtype=dt, device=DEV).normal_(generator=g)
        return dict(case=c, B=B, X=X, out=torch.empty((c["R"], n), dtype=dt, device=DEV))
    # features as the march forms them: the last eight values of smooth sequences over their RMS
    n = c["n"]
    t = torch.rand((n, 2), device=DEV, generator=g) * 6.0
    a = torch.randn((n, 2), device=DEV, generator=g)
    at = lambda k: a[:, 0] * torch.sin(t[:, 0] - 0.2 * k) + a[:, 1] * torch.cos(t[:, 1] - 0.35 * k)  # noqa: E731
    X = torch.stack([at(k) for k in range(1, 9)], dim=1).contiguous()
    Y = (at(0) - at(1)).contiguous()
    P = torch.zeros(4801, device=DEV)
    P[:512].uniform_(-8 ** -0.5, 8 ** -0.5, generator=g)
    P[576:4672].uniform_(-0.125, 0.125, generator=g)
    P[4736:4800].uniform_(-0.125, 0.125, generator=g)
    return dict(case=c, X=X, Y=Y, P=P, seed=seed)


def run(state):
    c = state["case"]
    if c["kind"] == "assemble":
        s = Solver(state["V"], state["F"], dt=c["dt"], nt=c["nt"], alpha=c["alpha"], precision=c["prec"], R=c["R"]).assemble()
        s.march(state["pw"], state["out"])
        s.close()
        return state["out"]
    if c["kind"] == "march":
        s = state["s"]
        _plan(s, c)
        s.set_excitation(state["pw"])
        s.step(c["nt"], state["out"])
        if c["ndir"]:
            return {"currents": state["out"], "far": s.far_field(state["out"], 1.5, state["rhat"])}
        return state["out"]
    if c["kind"] == "batch":
        for s, pw in zip(state["ss"], state["pw"]):
            s.set_excitation(pw)
        state["b"].step(c["nt"], state["outs"])
        return state["outs"]
    if c["kind"] == "block_gemv":
        return block_gemv(state["B"], state["X"], out=state["out"])
    P = state["P"].clone()
    loss = mlp_train(P, state["X"], state["Y"], epochs=c["epochs"], batch=c["batch"], lr=1e-3, seed=state["seed"])
    return {"params": P, "loss": loss}


# ---------------------------------------------------------------- work and exact values
def work(case):
    c = case
    if c["kind"] == "assemble":
        ne, nc, K = _sizes(c)
        # inner points of the outer points' polar rules (about 90 per pair, 40 operations each), the
        # static pairs, the products that form T_k, four inverses; the matrices written once
        flops = (7 + 18) * nc * nc * 90.0 * 40 + 36 * nc * nc * 9 * 30.0 + K * (4.0 * ne ** 3 + 4.0 * ne * nc * nc) + 6.0 * ne ** 3
        return {"bytes": 8.0 * ((3 * K + 8) * ne * ne + K * nc * nc), "flops": flops}
    if c["kind"] in ("march", "batch"):
        tot = {"bytes": 0.0, "flops": 0.0}
        for m in [c] if c["kind"] == "march" else [dict(_member(t), prec="fp32", R=1, form="dense", ndir=0) for t in c["members"].split(",")]:
            ne, nc, K = _sizes(m)
            es = 8 if m["prec"] == "fp64" else 4
            if m["form"] == "factored":     # about eleven shell entries per pair of edges, four bytes of index each
                entries, byts = 11.0 * ne * ne + ne * (2 * ne + nc) + nc * nc, 11.0 * ne * ne * (4 + es) + es * (ne * (2 * ne + nc) + nc * nc)
            else:
                entries = (K + 2.0) * ne * ne + nc * nc
                byts = entries * es
            tot["flops"] += 2.0 * c["nt"] * m["R"] * entries + 400.0 * m["ndir"] * nc
            tot["bytes"] += byts + 1.0 * c["nt"] * m["R"] * ne * es
        return tot
    if c["kind"] == "block_gemv":
        n, es = c["n"], 4 if c["dtype"] == "float32" else 8
        return {"bytes": es * (c["nblk"] * (1.0 * n * n + c["R"] * n) + c["R"] * n), "flops": 2.0 * c["nblk"] * c["R"] * n * n}
    return {"bytes": 36.0 * c["n"] * c["epochs"] + 8 * 4801, "flops": c["epochs"] * c["n"] * 6.0 * 4672}


def _mt19937_64(seed, count):
    """The first values of the 64-bit Mersenne Twister (Nishimura and Matsumoto, 2000)."""
    m64, n = (1 << 64) - 1, 312
    mt = [seed & m64]
    for i in range(1, n):
        mt.append((6364136223846793005 * (mt[-1] ^ (mt[-1] >> 62)) + i) & m64)
    for i in range(n):
        x = (mt[i] & 0xFFFFFFFF80000000) | (mt[(i + 1) % n] & 0x7FFFFFFF)
        mt[i] = mt[(i + 156) % n] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
    out = []
    for x in mt[:count]:
        x ^= (x >> 29) & 0x5555555555555555
        x ^= (x << 17) & 0x71D67FFFEDA60000
        x ^= (x << 37) & 0xFFF7EEE000000000
        out.append(x ^ (x >> 43))
    return out


def exact(case, seed):
    """In 64 bits by plain torch; None for the marches, whose values rest on the assembled integrals."""
    c = case
    if c["kind"] == "block_gemv":
        st = prepare(c, seed)
        out = torch.zeros((c["R"], c["n"]), dtype=torch.float64, device=DEV)
        for q in range(c["nblk"]):
            out += st["X"][q].double() @ st["B"][q].double().T
        return out
    if c["kind"] != "mlp_train":
        return None
    st = prepare(c, seed)
    n, nb = c["n"], -(-c["n"] // c["batch"])
    X, Y, p = st["X"].double(), st["Y"].double(), st["P"].double()
    m1, m2, losses, step = torch.zeros_like(p), torch.zeros_like(p), [], 0
    for rot in [x % n for x in _mt19937_64(seed, c["epochs"])]:
        loss = 0.0
        for b in range(nb):
            cnt = min(c["batch"], n - b * c["batch"])
            at = (torch.arange(cnt, device=DEV) + rot + b * c["batch"]) % n
            x, y = X[at], Y[at]
            W1, b1, W2, b2, W3, b3 = p[:512].view(64, 8), p[512:576], p[576:4672].view(64, 64), p[4672:4736], p[4736:4800], p[4800]
            h1 = torch.tanh(x @ W1.T + b1)
            h2 = torch.tanh(h1 @ W2.T + b2)
            r = h2 @ W3 + b3 - y
            loss += 0.5 * float((r * r).mean())
            d = r / cnt
            d2 = d[:, None] * W3 * (1 - h2 * h2)
            d1 = (d2 @ W2) * (1 - h1 * h1)
            g = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), d @ h2, d.sum()[None]])
            step += 1
            m1 = 0.9 * m1 + 0.1 * g
            m2 = 0.999 * m2 + 0.001 * g * g
            p = p - 1e-3 * (m1 / (1 - 0.9 ** step)) / (torch.sqrt(m2 / (1 - 0.999 ** step)) + 1e-8)
        losses.append(loss / nb)
    return {"params": p, "loss": np.array(losses)}
