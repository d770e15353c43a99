"""The partial sums of K belong to the handle's workspace: a graph captured at one
orbital count replays correctly after builds at smaller counts (which can need
more splits), density builds and the setup of another molecule, and the two
spins of an unrestricted build, queued without a wait, equal single builds."""
import numpy as np
import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


def _c(m, nocc, seed):
    return torch.from_numpy(np.random.default_rng(seed).standard_normal((m.nao, nocc))).cuda() / m.nao**0.5


# mixed, nao 375: 104 orbitals give 25 splits of K, 82 give 26 (tests/test_k_split.py)
@pytest.mark.parametrize("precision,natom,big,small", [(dfjk.DFJK_MIXED, 25, 104, 82), (dfjk.DFJK_FP64, 9, 41, 17)])
def test_replay_after_smaller_builds(precision, natom, big, small):
    m, other = I.molecule(natom, seed=1000 + natom), I.molecule(natom, seed=1100 + natom)
    h = dfjk.Handle(m, precision=precision)
    C = _c(m, big, 1)
    J, K, _, _ = h.build(C)
    J1, K1 = torch.empty_like(J), torch.empty_like(K)
    E = torch.empty((2, 1), dtype=torch.float64, device="cuda")
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        dfjk.build_batch([h], [C], Js=[J1[0]], Ks=[K1[0]], E=E, nstreams=1, stream=s)
    h.build(_c(m, small, 2))
    D = torch.randn(m.nao, m.nao, dtype=torch.float64, device="cuda")
    h.build_density(D + D.T)
    f = dfjk.Handle(other, precision=precision)
    Co = _c(other, big, 3)
    Jo, Ko, _, _ = f.build(Co)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(J, J1) and torch.equal(K, K1)
    Jp, Kp, _, _ = f.build(Co)  # the replay left the other molecule's buffers alone
    assert torch.equal(Jo, Jp) and torch.equal(Ko, Kp)
    f.close()
    h.close()


def test_unrestricted_build_with_more_splits_in_the_second_spin():
    m = I.molecule(25, seed=1025)
    h = dfjk.Handle(m, precision=dfjk.DFJK_MIXED)
    Ca, Cb = _c(m, 104, 4), _c(m, 82, 5)
    Ka, Kb = h.build(Ca)[1][0], h.build(Cb)[1][0]
    f = dfjk.Handle(m, precision=dfjk.DFJK_MIXED)
    _, Kua, Kub, _ = f.build_uks(Ca, Cb)[:4]
    assert torch.equal(Ka, Kua) and torch.equal(Kb, Kub)
    f.close()
    h.close()
