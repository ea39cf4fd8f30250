"""GPU: device work of a handle is ordered with its stream, also where a batch runs it on another one.

A fill of the output buffers is queued behind a slow kernel on the stream that the caller uses (the
handle's own opts.stream, or the legacy default stream for a handle without one); a call made right
after must write its currents after that fill."""
import pytest

from synth import excitation, meshes

pytestmark = pytest.mark.gpu

NT = 20
SLOW = 100_000_000      # clock cycles that the queued kernel takes (about 50 ms)


@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("precisions", [("fp32", "fp32"), ("fp64", "fp32")])      # persistent form, graph branches
def test_batch_waits_for_the_members_streams(own, precisions):
    import torch
    from paper_2312_06367_gb300 import Batch, Solver
    mesh = [meshes.icosphere(0), meshes.torus(1.0, 0.4, 5, 3)]
    pw = excitation.single(t0=3.0, sigma=0.8)
    streams = [torch.cuda.default_stream() if own else torch.cuda.Stream() for _ in mesh]
    ss = [Solver(*m, dt=0.4, nt=NT, precision=p, stream=None if own else st.cuda_stream).assemble()
          for m, p, st in zip(mesh, precisions, streams)]
    outs = [torch.zeros((NT, 1, s.ne), dtype=s.dtype, device="cuda") for s in ss]
    refs = [torch.zeros_like(o) for o in outs]
    torch.cuda.synchronize()
    for s, ref in zip(ss, refs):
        s.march(pw, ref)
        s.set_excitation(pw)
    b = Batch(ss)
    torch.cuda.synchronize()
    for st, o in zip(streams, outs):
        with torch.cuda.stream(st):
            torch.cuda._sleep(SLOW)
            o.fill_(7.0)
    b.step(NT, outs)
    torch.cuda.synchronize()
    b.close()
    for o, ref in zip(outs, refs):
        assert torch.equal(o, ref)


@pytest.mark.parametrize("precision,R,kw", [("fp64", 1, {}), ("fp32", 3, {"solver": "gmres", "guess": "extrap"}), ("fp16x3", 64, {})])
def test_plan_state_does_not_wait_for_the_legacy_stream(precision, R, kw):
    """Plan, solver state and their resets are on the handle's stream: work pending on the legacy stream
    meanwhile neither delays them into a running march nor leaves them out."""
    import torch
    from paper_2312_06367_gb300 import Solver
    V, F = meshes.icosphere(1)
    pw = excitation.fibonacci_batch(R, seed=3, t0=3.0, sigma=0.8)
    st = torch.cuda.Stream()

    def march(busy):
        def hold():
            if busy:
                with torch.cuda.stream(torch.cuda.default_stream()):
                    torch.cuda._sleep(SLOW)
        out = torch.zeros((NT, R, 120), dtype=torch.float64 if precision == "fp64" else torch.float32, device="cuda")
        s = Solver(V, F, dt=0.4, nt=NT, precision=precision, R=R, stream=st.cuda_stream)
        torch.cuda.synchronize()
        s.assemble()
        if kw:
            hold()
            s.set_solver(kw["solver"], kw["guess"], 1e-9)
        else:
            hold()
            s.replan(precision, R)
        s.set_excitation(pw)
        s.step(7, out[:7])
        hold()
        s.set_excitation(pw)
        s.step(NT, out)
        torch.cuda.synchronize()
        return out

    ref = march(False)
    assert torch.isfinite(ref).all()
    # (the FP64 assembly adds with atomics, so two assemblies agree to rounding only)
    assert float((march(True) - ref).double().norm() / ref.double().norm()) < 1e-5
