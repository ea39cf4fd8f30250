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
