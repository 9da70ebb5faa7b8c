"""Which transforms a WGS loop runs on. An iteration divides by the spots'
amplitudes: where one passes near zero, the loop multiplies the transforms'
rounding by 100 and more, so that loops of small holograms return what they
returned only on the same kernels. Below side 560 those are the ones of
variants 1 and 2 (FMA pipe for few spots, tensor cores for many), whatever a
single transform of the same handle runs on: every result is compared bit for
bit with that variant's, alone and as a standalone member of a batch.
"""
import pytest

torch = pytest.importorskip("torch")

from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu

LOW = [2, 3, 4, 5, 6]
CASES = [  # (nx, ny, N, noll, variant of the loop): 1 below 64 spots, 2 from 256
    (384, 400, 50, LOW, 1),
    (512, 512, 63, LOW, 1),
    (512, 512, 260, LOW, 2),
    (233, 559, 300, LOW, 2),
    (450, 470, 280, list(range(2, 12)), 2),
]


def _state(p):
    t = torch.from_numpy(p.target).cuda()
    return torch.from_numpy(p.phase0).cuda().clone(), t.clone(), t


def _loop(p, variant):
    from paper_2505_08777_gb300 import Hologram
    h = Hologram(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), noll=p.noll)
    h.set_variant(variant)
    ph, w, t = _state(p)
    E, met = h.wgs(ph, w, t, 4)
    assert h.graph_kernels(4) == h.wgs_launches(4)
    h.check()
    return ph, w, E, met


def test_small_loops_stay_on_their_kernels():
    from paper_2505_08777_gb300 import Batch
    ps = [random_problem(900 + k, nx, ny, N, noll) for k, (nx, ny, N, noll, _) in enumerate(CASES)]
    own = []
    for p, c in zip(ps, CASES):
        auto = _loop(p, 0)
        assert all(torch.equal(a, b) for a, b in zip(auto, _loop(p, c[4]))), c
        own.append(auto)
    b = Batch([(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), p.noll) for p in ps], solo_terms=0)
    states = [_state(p) for p in ps]
    met = b.wgs([s[0] for s in states], [s[1] for s in states], [s[2] for s in states], 4)
    assert b.graph_kernels(4) == b.launches(4)
    for k, (ph, w, _, m) in enumerate(own):
        assert torch.equal(states[k][0], ph) and torch.equal(states[k][1], w) and torch.equal(met[k], m), CASES[k]
