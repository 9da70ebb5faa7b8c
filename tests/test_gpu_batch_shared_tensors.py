"""A batch whose members share a phase or weight tensor ends with the last
member's values in it, whatever the sizes: every member reads the tensor as it
was before the call, and the results are written in the members' order."""
import pytest

torch = pytest.importorskip("torch")

from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,N,count", [(512, 512, 40, 6), (64, 33, 7, 50), (256, 256, 3000, 3)])
def test_last_member_wins(nx, ny, N, count):
    from paper_2505_08777_gb300 import Batch
    ps = [random_problem(300 + k, nx, ny, N, list(range(2, 12))) for k in range(count)]
    b = Batch([(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), p.noll) for p in ps])
    ph0, t = torch.from_numpy(ps[0].phase0).cuda(), torch.ones(N, device="cuda")
    ph, w = [ph0.clone() for _ in ps], [t.clone() for _ in ps]
    met = b.wgs(ph, w, [t] * count, 2)
    for _ in range(3):
        one, wone = ph0.clone(), t.clone()
        met1 = b.wgs([one] * count, [wone] * count, [t] * count, 2)
        assert torch.equal(one, ph[-1]) and torch.equal(wone, w[-1]) and torch.equal(met1, met)
