"""Product-sum decoding with four lanes a check at its largest sizes (97 to 128
columns, which fill its variable passes, and up to 128 checks in 16 rounds) and
with learned weights, against the oracle and the weighted reference."""
import numpy as np
import pytest
import scipy.sparse as sp

import bpdc_inputs as bi
import parity
from bpdc_inputs.codes import Problem, _csr
from bpdc_inputs.sampler import sample_shots
from oracle import weighted_bp
from parity import to_dev

pytestmark = pytest.mark.gpu


def _problem(M, N, seed):
    """Every check has 1 to 4 edges, every column 1 or 2."""
    rng = np.random.default_rng(seed)
    H = np.zeros((M, N), np.uint8)
    for j in range(N):
        H[j % M, j] = 1
    for j in rng.permutation(N):
        free = np.nonzero((H.sum(1) < 4) & (H[:, j] == 0))[0]
        if len(free) and rng.random() < 0.8:
            H[rng.choice(free), j] = 1
    D = np.zeros((N // 4, N), np.uint8)
    for r in range(N // 4):
        D[r, rng.choice(N, 5, replace=False)] = 1
    L = rng.random((2, N)) < 0.4
    return Problem(f"largest{M}", _csr(sp.csr_matrix(H)), _csr(sp.csr_matrix(D)), _csr(L), rng.uniform(0.02, 0.2, N))


@pytest.mark.parametrize("M,N", [(33, 97), (57, 128), (64, 100), (65, 128), (127, 127), (128, 128)])
def test_largest_sizes_match_the_oracle(M, N, oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    P = _problem(M, N, 1000 * M + N)
    w = np.diff(P.H.tocsr().indptr)
    assert w.min() >= 1 and w.max() == 4 and P.H.shape == (M, N) and (N + 31) // 32 == 4
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


@pytest.mark.parametrize("d", [3, 5])
def test_learned_weights_match_the_reference(d):
    """Plain BP with learned weights: the first iteration whose decision
    reproduces the syndrome and the posterior there, on shots whose reference
    posteriors stay away from 0 up to it."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    P, T = bi.surface_problem(d, 0.08), 6
    W = np.random.default_rng(d).uniform(0.7, 1.3, size=(2, T, P.E))
    _, s, _ = sample_shots(P, 9, 0, 300)
    g = pkg.Graph.from_problem(P, pkg.Options(variant=1, max_iter=T, dc_enable=0))
    assert g.info["kernel_id"] == 11
    g.set_weights(torch.tensor(W, dtype=torch.float32), clip=20.0)
    assert g.info["kernel_id"] == 11
    out = g.decode(to_dev(s), 0, posterior=True)
    again = g.decode(to_dev(s), 0)
    assert all(torch.equal(out[k], again[k]) for k in again)
    it, st = out["iterations"].cpu().numpy() & 0xFFFF, out["status"].cpu().numpy()
    post = out["posterior_llr"].cpu().numpy().astype(np.float64)
    rp = weighted_bp.forward(P.H, P.priors, s, torch.tensor(W.astype(np.float32)).double()).numpy()
    H = P.H.toarray().astype(np.int64)
    lam = np.log((1 - P.priors) / P.priors)
    checked = 0
    for b in range(len(s)):
        hist = [lam] + list(rp[b])
        conv = [t for t in range(T + 1) if (((H @ (hist[t] <= 0)) % 2) == s[b]).all()]
        t = conv[0] if conv else T
        if any(np.abs(h).min() < 1e-3 for h in hist[1:t + 1]):
            continue
        checked += 1
        assert st[b] == (0 if conv else 2) and it[b] == t, b
        assert (np.abs(post[b] - hist[t]) / np.maximum(np.abs(hist[t]), 1.0)).max() < 1e-4
    assert checked > 250
