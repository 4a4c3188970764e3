"""Product-sum decoding with four lanes a check, at the edges of its rounds of
eight checks: one check, a round less or more by one, the most checks; rows of 1
to 4 edges, columns of weight 1 and 2, uneven priors; against the oracle by the rules
of parity.py."""
import numpy as np
import pytest
import scipy.sparse as sp

import parity
from bpdc_inputs.codes import Problem, _csr
from bpdc_inputs.sampler import sample_shots
from parity import to_dev

pytestmark = pytest.mark.gpu


def _problem(M, seed):
    rng = np.random.default_rng(seed)
    ends = np.repeat(np.arange(M), rng.integers(1, 5, M))   # row weights 1 .. 4
    rng.shuffle(ends)
    cols = []
    while len(ends):
        pair = len(ends) > 1 and ends[0] != ends[1] and rng.random() < 0.8 and len(cols) < 127
        cols.append(ends[:2] if pair else ends[:1])
        ends = ends[2 if pair else 1:]
    cols = cols[:128]
    N = len(cols)
    H = sp.lil_matrix((M, N), dtype=np.uint8)
    for j, c in enumerate(cols):
        H[c, j] = 1
    D = sp.lil_matrix((max(1, N // 4), N), dtype=np.uint8)
    for r in range(D.shape[0]):
        D[r, rng.choice(N, min(N, 5), replace=False)] = 1
    L = rng.random((2, N)) < 0.4
    return Problem(f"rounds{M}", _csr(H), _csr(D), _csr(L), rng.uniform(0.02, 0.2, N))


@pytest.mark.parametrize("M", [1, 2, 7, 8, 9, 31, 33, 56])
def test_rounds_of_checks_match_the_oracle(M, oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    P = _problem(M, 100 + M)
    _, s, o = sample_shots(P, 5, 0, 400)
    g = pkg.Graph.from_problem(P, pkg.Options(variant=1, max_iter=12, dc_prior=M % 2))
    assert g.info["kernel_id"] == 11
    out = g.decode(to_dev(s), 0, obs_true=to_dev(o), posterior=True)
    plain = g.decode(to_dev(s), 0, obs_true=to_dev(o), persistent=False)
    for k in ("corrections", "status", "logical_flips", "iterations"):
        assert bool((out[k] == plain[k]).all()), k
    opts = oracle_mod.Options(variant=1, max_iter=12, dc_prior=M % 2)
    rep = parity.compare(oracle_mod, P, s, 0, opts, parity.gpu_outcome(P, out), obs=o)
    assert rep["unmatched_well"] == 0, parity.summary(rep)
    assert rep["posterior"]["failed"] == 0 and rep["posterior"]["inf_mismatch"] == 0, rep["posterior"]
