"""bta_assemble takes blocks on 8-byte boundaries, as the factor does."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(8, 8), (7, 5)])
@pytest.mark.parametrize("which", [0, 1])
def test_assemble_into_unaligned_blocks(nx, ny, which):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_06392_gb300 import build
    build.build()
    import paper_2605_06392_gb300 as P
    prob = workloads.make_problem("st_tiny", nx=nx, ny=ny, nt=3)
    m = P.InlaModel(prob)
    a = m.a if which else 0
    out = []
    for off in (0, 1):
        q = P.BtaMatrix(m.n, m.b, a, m.ld)
        guards = []
        for name in ("D", "B"):
            t = getattr(q, name)
            buf = torch.full((t.numel() + 2,), 7.0, dtype=torch.float64, device="cuda")
            setattr(q, name, buf[off:off + t.numel()].view(t.shape))
            setattr(q.desc, name, getattr(q, name).data_ptr())
            guards.append((buf[:off], buf[off + t.numel():]))
        P.bta_assemble(m, prob.theta, which, q)
        torch.cuda.synchronize()
        assert all(bool((part == 7.0).all()) for pair in guards for part in pair)
        out.append((q.D.cpu(), q.B.cpu()))
    m.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
