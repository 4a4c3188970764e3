"""The GPU shot sampler at the edges of its forms: a shot in registers (up
to 256 columns), columns listed in shared memory by a warp (up to 1024) or by a
block per shot; no, one, few and many logical words; short and odd batches.
Every word equals the CPU sampler's."""
import numpy as np
import pytest
import scipy.sparse as sp

from bpdc_inputs.codes import Problem, _csr
from bpdc_inputs.sampler import sample_shots
from parity import from_dev

pytestmark = pytest.mark.gpu


def _problem(N, K, seed):
    """Columns of weight 2 on rows of weight <= 8, uneven priors."""
    rng = np.random.default_rng(seed)
    M = max(2, (N + 3) // 4)
    first = np.arange(N) % M
    H = sp.csr_matrix((np.ones(2 * N, np.uint8), (np.r_[first, (first + 1) % M], np.r_[np.arange(N), np.arange(N)])),
                      shape=(M, N))
    L = _csr(rng.random((K, N)) < 0.3) if K else sp.csr_matrix((0, N), dtype=np.uint8)
    return Problem(f"n{N}", _csr(H), sp.csr_matrix((0, N), dtype=np.uint8), L, rng.uniform(0.001, 0.5, N))


@pytest.mark.parametrize("N,K,B", [(8, 0, 1), (32, 1, 7), (33, 33, 100), (255, 3, 9), (256, 256, 33), (250, 300, 17),
                                   (257, 1, 65), (1000, 40, 5), (1024, 300, 31), (1025, 2, 3), (1500, 100, 1300),
                                   (2500, 257, 21), (200, 1200, 11)])
def test_sampler_matches_cpu(N, K, B):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    P = _problem(N, K, N + K)
    g = pkg.Graph.from_problem(P)
    off = (1 << 40) + 12345
    syn, obs, err = g.sample(B, 99, off, errors=True)
    e, s, o = sample_shots(P, 99, off, B)
    assert (from_dev(err, P.N) == e).all()
    assert (from_dev(syn, P.M) == s).all()
    if K:
        assert (from_dev(obs, P.K) == o).all()
    assert torch.equal(g.sample(B, 99, off)[0], syn)
