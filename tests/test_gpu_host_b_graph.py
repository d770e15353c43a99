"""A build of a handle with B in host memory, captured in a graph, replays after calls
that stage larger pieces of B (density build, gradient) and after another
molecule's setup, and equals the direct build, bit for bit."""
import numpy as np
import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


@pytest.mark.parametrize("precision", [dfjk.DFJK_FP64, dfjk.DFJK_MIXED])
def test_replay_after_other_calls(precision, tmp_path):
    table = tmp_path / "tune.txt"
    table.write_text("1 100000 16 8 64 8\n")  # 8 MB of work buffers: chunks of 128 rows in the build
    m = I.molecule(9, seed=1009)
    h = dfjk.Handle(m, precision=precision, b_on_host=True, tune_table=str(table))
    rng = np.random.default_rng(9)
    C = torch.from_numpy(rng.standard_normal((m.nao, 27))).cuda()
    J, K, _, _ = h.build(C)
    J1, K1 = torch.empty_like(J), torch.empty_like(K)
    E = torch.empty((2, 1), dtype=torch.float64, device="cuda")
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        dfjk.build_batch([h], [C], Js=[J1[0]], Ks=[K1[0]], E=E, nstreams=1, stream=s)
    h.build_density(C @ C.T)
    h.jk_gradient(C, 1.0, -0.5)
    f = dfjk.Handle(I.molecule(9, seed=1109), precision=precision)
    T = f.build(C)[1]
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(J, J1) and torch.equal(K, K1)
    assert torch.equal(T, f.build(C)[1])
    f.close()
    h.close()
