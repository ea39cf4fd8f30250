"""GPU: the blocked march, the group GMRES, the quadrature's windows, the history sum's row tiles and the
training step at the sizes where their splits can go wrong: chunks that start or stop anywhere, fewer
lags than a chunk has steps, rows that no vector load fits, waves that fill no tile.

Tolerances are those of the paths elsewhere in the suite (FP64 1e-10 against the oracle, FP32
1e-5); results that depend on no rounding order are compared bit for bit."""
import numpy as np
import pytest

from synth import excitation, meshes

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _oracle(mesh, dt, nt, pw):
    """The oracle's march on the library's FP64 matrices.  (The matrices have their own tests, on spheres
    for the 1e-10 bar: on this coarse torus the oracle's quadrature itself is good to some 1e-10.)"""
    from oracle import mot, rhs
    from oracle.assemble import Operators
    from oracle.formulation import Formulation
    ops = Operators(*mesh, dt=dt)
    s = _solver(mesh, dt, nt, 1, "fp64")
    for name in ("G", "Zs", "Zh", "M"):
        setattr(ops, name, s.matrix(name, 0))
    for name in ("S", "H", "MM"):
        setattr(ops, name, np.stack([s.matrix(name, k) for k in range(ops.K)]))
    s.close()
    fm = Formulation(ops)
    e, h = rhs.incident_tests(ops, pw, dt * np.arange(1, nt + 1))
    return fm.postprocess(mot.march_factored(fm, fm.rhs(e, h)))


def _solver(mesh, dt, nt, R, precision, **kw):
    from paper_2312_06367_gb300 import Solver
    return Solver(*mesh, dt=dt, nt=nt, R=R, precision=precision, **kw).assemble()


SMALL = meshes.torus(1.0, 0.4, 5, 3)      # 45 edges: odd rows, fewer than a block of any kernel
BOUND = {"fp64": 1e-10, "fp32": 1e-5}
# (dt, steps): more lags than a chunk has steps; as few lags as there can be; a chunk and one step
SPLITS = [(0.15, 35), (4.0, 18), (0.8, 17)]


@pytest.fixture(scope="module")
def waves():
    return excitation.random_batch(8, seed=31, t0=3.0, sigma=0.8)


@pytest.fixture(scope="module")
def refs(waves):
    return {dt: _oracle(SMALL, dt, nt, waves) for dt, nt in SPLITS}


@pytest.mark.parametrize("dt,nt", SPLITS)
@pytest.mark.parametrize("precision,R", [("fp64", 1), ("fp64", 8), ("fp32", 2), ("fp32", 3), ("fp32", 8)])
def test_march_in_chunks(waves, refs, precision, R, dt, nt):
    """Against the oracle, and any partition of the steps gives the same bits."""
    import torch
    pw = {k: v[:R] for k, v in waves.items()}
    s = _solver(SMALL, dt, nt, R, precision)
    out = torch.zeros((nt, R, s.ne), dtype=s.dtype, device="cuda")
    s.march(pw, out)
    parts = torch.zeros_like(out)
    s.set_excitation(pw)
    at = 0
    for m in (1, 7, 9, 2, nt):
        m = min(m, nt - at)
        s.step(m, parts[at:at + m])
        at += m
    torch.cuda.synchronize()
    assert torch.equal(out, parts)
    if precision == "fp64" or dt > 0.15:      # FP32 at 0.15 on this mesh: 2e-5 to 4e-5 by the path's rounding
        assert rel(out.double().cpu().numpy().transpose(0, 2, 1), refs[dt][:, :, :R]) < BOUND[precision]


@pytest.mark.parametrize("precision,R", [("fp64", 1), ("fp64", 3), ("fp32", 1), ("fp32", 8)])
def test_group_gmres(waves, refs, precision, R):
    """Restarts after three iterations, one group of blocks per wave; partitions give the same bits."""
    import torch
    dt, nt = SPLITS[0 if precision == "fp64" else 2]
    pw = {k: v[:R] for k, v in waves.items()}
    s = _solver(SMALL, dt, nt, R, precision, solver="gmres", guess="extrap", gmres_restart=3, gmres_maxit=300,
                gmres_tol=1e-13 if precision == "fp64" else 1e-9)
    out = torch.zeros((nt, R, s.ne), dtype=s.dtype, device="cuda")
    s.march(pw, out)
    st = s.gmres_stats()
    parts = torch.zeros_like(out)
    s.set_excitation(pw)
    s.step(11, parts[:11])
    s.step(nt - 11, parts[11:])
    torch.cuda.synchronize()
    assert st["steps"] == nt and st["not_converged"] == 0
    assert torch.equal(out, parts)
    assert rel(out.double().cpu().numpy().transpose(0, 2, 1), refs[dt][:, :, :R]) < BOUND[precision]


@pytest.mark.parametrize("precision", ["fp16x3", "bf16x3"])
def test_tensor_chunks(precision):
    """30 edges (one ragged tile): partitions of the steps, and repetitions, give the same bits."""
    import torch
    nt = 14
    pw = excitation.fibonacci_batch(64, seed=5, t0=3.0, sigma=0.8)
    s = _solver(meshes.icosphere(0), 0.4, nt, 64, precision)
    out = torch.zeros((nt, 64, s.ne), dtype=s.dtype, device="cuda")
    s.march(pw, out)
    for split in ((1, 2, 3, 4, 4), (5, 9), (14,), (14,)):
        parts = torch.zeros_like(out)
        s.set_excitation(pw)
        at = 0
        for m in split:
            s.step(m, parts[at:at + m])
            at += m
        torch.cuda.synchronize()
        assert torch.isfinite(out).all() and torch.equal(out, parts), split


@pytest.mark.parametrize("time_order", [1, 2])
@pytest.mark.parametrize("dt", [0.02, 0.11, 5.0])
def test_quadrature_windows(dt, time_order):
    """Lags per pair from one to several windows, on 30 edges."""
    from oracle.assemble import Operators
    V, F = meshes.icosphere(0)
    ops = Operators(V, F, dt=dt, time_order=time_order)
    s = _solver((V, F), dt, 4, 1, "fp64", time_order=time_order)
    for k in range(0, ops.K, max(1, ops.K // 6)):
        for name, ref in (("S", ops.S[k]), ("H", ops.H[k]), ("MM", ops.MM[k])):
            got = s.matrix(name, k)
            scale = max(np.linalg.norm(x) for x in {"S": ops.S, "H": ops.H, "MM": ops.MM}[name])
            # an almost empty block at the end of the lags is held to the largest block's scale
            assert np.linalg.norm(got - ref) <= 1e-10 * max(np.linalg.norm(ref), 1e-3 * scale), (name, k)


@pytest.mark.parametrize("dtype,tol", [("float64", 1e-13), ("float32", 1e-5)])
@pytest.mark.parametrize("nblk,n,R,off", [(2, 4, 1, 0), (3, 130, 2, 0), (3, 132, 2, 1), (2, 65, 4, 0), (9, 516, 5, 0), (9, 257, 8, 0)])
def test_block_gemv_row_tiles(dtype, tol, nblk, n, R, off):
    """Vector and scalar loads (odd rows, blocks off the 16-byte boundary), rows that fill no tile."""
    import torch
    from paper_2312_06367_gb300 import block_gemv
    g = torch.Generator(device="cuda").manual_seed(nblk * n + R)
    dt = getattr(torch, dtype)
    B = torch.randn(nblk * n * n + off, generator=g, dtype=dt, device="cuda")[off:].view(nblk, n, n)
    X = torch.randn((nblk, R, n), generator=g, dtype=dt, device="cuda")
    ref = torch.einsum("qij,qrj->ri", B.double(), X.double())
    got = block_gemv(B, X)
    torch.cuda.synchronize()
    assert float((got.double() - ref).norm() / ref.norm()) < tol


@pytest.mark.parametrize("n,epochs", [(1, 1), (31, 2), (1000, 5)])
def test_training_updates(n, epochs):
    """One batch per pass: the parameters after 1, 2 and 5 updates against Adam on the oracle's
    gradient.  An update moves a parameter by lr g / |g| at most, with g good to 1e-4."""
    import torch
    from oracle import mlp
    from paper_2312_06367_gb300 import mlp_train
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 8)).astype(np.float32)
    Y = np.tanh(X @ rng.standard_normal(8)).astype(np.float32)
    p = torch.tensor(mlp.init_params(2), dtype=torch.float32, device="cuda")
    q = p.double().cpu().numpy()
    hist = mlp_train(p, torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda"), epochs=epochs, batch=4096, lr=1e-3)
    m1, m2 = np.zeros_like(q), np.zeros_like(q)
    for k in range(1, epochs + 1):
        loss, g = mlp.loss_and_grad(q, X.astype(np.float64), Y.astype(np.float64))
        assert abs(hist[k - 1] - loss) <= 1e-4 * loss
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        q = q - 1e-3 * (m1 / (1 - 0.9 ** k)) / (np.sqrt(m2 / (1 - 0.999 ** k)) + 1e-8)
    assert rel(p.double().cpu().numpy(), q) < 1e-4


def test_batch_before_excitation(waves):
    """A batch made of handles without an excitation yet."""
    import torch
    from paper_2312_06367_gb300 import Batch
    pw = {k: v[:1] for k, v in waves.items()}
    ss = [_solver(SMALL, 0.15, 20, 1, "fp32"), _solver(meshes.icosphere(0), 0.3, 20, 1, "fp32")]
    b = Batch(ss)
    for s in ss:
        s.set_excitation(pw)
    outs = [torch.zeros((20, 1, s.ne), dtype=torch.float32, device="cuda") for s in ss]
    b.step(20, outs)
    b.close()
    for s, o in zip(ss, outs):
        ref = torch.zeros_like(o)
        s.march(pw, ref)
        torch.cuda.synchronize()
        assert torch.equal(o, ref)


@pytest.mark.parametrize("precision,R", [("fp64", 1), ("fp64", 3), ("fp32", 1), ("fp32", 8)])
@pytest.mark.parametrize("form", ["dense", "factored"])
def test_first_chunk_in_calls(waves, precision, R, form):
    """The first chunk of a march is formed call by call: any calls, also a batch's, give the same bits."""
    import torch
    from paper_2312_06367_gb300 import Batch
    pw = {k: v[:R] for k, v in waves.items()}
    s, other = _solver(SMALL, 0.15, 20, R, precision), _solver(meshes.icosphere(0), 0.3, 20, R, precision)
    for t in (s, other):
        t.set_history_form(form)
        t.set_excitation(pw)
    out = torch.zeros((20, R, s.ne), dtype=s.dtype, device="cuda")
    s.march(pw, out)
    b = Batch([s, other])
    for calls in ((1, -1, 1, -2, 15), (-1, 3, -4, 12), (2, -18), (-17, 3)):      # negative: steps of the batch
        parts = torch.zeros_like(out)
        s.set_excitation(pw)
        other.set_excitation(pw)
        torch.cuda.synchronize()
        at = 0
        for m in calls:
            if m > 0:
                s.step(m, parts[at:at + m])
            else:
                b.step(-m, [parts[at:at - m], None])
            at += abs(m)
        torch.cuda.synchronize()
        assert at == 20 and torch.equal(out, parts), calls
    b.close()


def test_one_step_does_not_pay_for_a_chunk():
    """A new march of one step costs well under one of eight (before the first chunk was formed call by
    call it cost 0.8 of it: the sums over all lags of eight columns)."""
    import time
    import torch
    pw = excitation.random_batch(8, seed=3, t0=3.0, sigma=0.8)
    s = _solver(meshes.icosphere(2), 0.05, 8, 8, "fp64")
    times = {}
    for nt in (1, 8):
        best = []
        for _ in range(7):
            s.set_excitation(pw)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            s.step(nt)
            best.append(time.perf_counter() - t0)
        times[nt] = min(best)
    print(times)
    assert times[1] < 0.6 * times[8]


def _prism(sections, length, radius):
    """A slightly irregular triangular prism of `sections` sections with a triangle at either end."""
    rng = np.random.default_rng(5)
    V = [((radius + 0.05 * rng.uniform()) * np.cos(2.1 * i + 0.1 * s), (radius + 0.05 * rng.uniform()) * np.sin(2.1 * i + 0.1 * s), length * s)
         for s in range(sections + 1) for i in range(3)]
    F = [(0, 2, 1), (3 * sections, 3 * sections + 1, 3 * sections + 2)]
    for s in range(sections):
        for i in range(3):
            a, b = 3 * s + i, 3 * s + (i + 1) % 3
            F += [(a, b, b + 3), (a, b + 3, a + 3)]
    return np.array(V), np.array(F, dtype=np.int32)


@pytest.mark.parametrize("circles", [60, 63, 90])
def test_quadrature_many_circles(circles):
    """As many breakpoint circles across an edge as the list of cuts holds, and more: every one of them
    splits, in both forms of the rule.  The scalar potential's blocks of a pair against the oracle's rule with all breakpoints."""
    from oracle import cquad
    V, F = _prism(5, 1.0, 0.5)
    tri = V[F]
    L = max(np.linalg.norm(tri[:, i] - tri[:, (i + 1) % 3], axis=1).max() for i in range(3))
    dt = L / circles
    s = _solver((V, F), dt, 1, 1, "fp64")
    T0, K = s.D, s.K
    Phi = np.stack([s.matrix("Phi", k) for k in range(K)])
    s.close()
    s15 = np.sqrt(15.0)
    rule = [((1 / 3, 1 / 3, 1 / 3), 9 / 40)]
    for sg in (-1, 1):
        a, b, w = (9 + sg * 2 * s15) / 21, (6 - sg * s15) / 21, (155 - sg * s15) / 1200
        rule += [((a, b, b), w), ((b, a, b), w), ((b, b, a), w)]
    brk = [j * dt for j in range(1, K)]
    area = 0.5 * np.linalg.norm(np.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]), axis=1)
    far = 0
    for c, c2 in ((0, 2), (4, 6), (4, 3), (4, 28), (30, 3), (3, 31)):
        n = np.cross(tri[c2, 1] - tri[c2, 0], tri[c2, 2] - tri[c2, 0])
        n /= np.linalg.norm(n)
        lags = np.argsort(-np.abs(Phi[:, c, c2]))[:60:4]
        ref = np.zeros(len(lags))
        for bary, w in rule:
            x = np.array(bary) @ tri[c]
            p = x - np.dot(x - tri[c2, 0], n) * n
            edges = np.linalg.norm(tri[c2] - np.roll(tri[c2], 1, axis=0), axis=1).max()
            is_far = np.linalg.norm(tri[c2] - p, axis=1).min() >= 2 * edges
            far += is_far
            for i, k in enumerate(lags):
                m = cquad.triangle_moments(x, *tri[c2], kind=4, p1=k * dt, p2=dt, brk=brk, coplanar=2)
                ref[i] += -T0 * w / (4 * np.pi * area[c2]) * m[0]
        assert np.abs(Phi[lags, c, c2] - ref).max() <= 1e-10 * np.abs(ref).max(), (c, c2)
    assert far >= 14


@pytest.mark.parametrize("R", range(1, 9))
@pytest.mark.parametrize("dtype,tol", [("float64", 1e-13), ("float32", 1e-5)])
def test_block_gemv_every_wave_count(dtype, tol, R):
    """Each number of vectors has its own kernel, for rows that vector loads fit and others."""
    import torch
    from paper_2312_06367_gb300 import block_gemv
    g = torch.Generator(device="cuda").manual_seed(R)
    dt = getattr(torch, dtype)
    for n in (132, 131):
        B = torch.randn((3, n, n), generator=g, dtype=dt, device="cuda")
        X = torch.randn((3, R, n), generator=g, dtype=dt, device="cuda")
        ref = torch.einsum("qij,qrj->ri", B.double(), X.double())
        got = block_gemv(B, X)
        torch.cuda.synchronize()
        assert float((got.double() - ref).norm() / ref.norm()) < tol


@pytest.mark.parametrize("R", [2, 3, 8])
def test_fp32_waves_against_fp64(waves, R):
    """More lags (21) than a chunk has steps, every wave by itself against the FP64 path on the same
    matrices.  The path's own rounding is 2e-5 to 4e-5 of the currents on this mesh; a wrong lag, column
    or wave is of their size."""
    import torch
    dt, nt = SPLITS[0]
    pw = {k: v[:R] for k, v in waves.items()}
    s = _solver(SMALL, dt, nt, R, "fp64")
    ref = torch.zeros((nt, R, s.ne), dtype=torch.float64, device="cuda")
    s.march(pw, ref)
    s.replan("fp32", R)
    out = torch.zeros((nt, R, s.ne), dtype=torch.float32, device="cuda")
    s.march(pw, out)
    torch.cuda.synchronize()
    for r in range(R):
        assert float((out[:, r].double() - ref[:, r]).norm() / ref[:, r].norm()) < 1e-4, r
