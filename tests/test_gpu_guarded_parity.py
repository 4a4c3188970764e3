"""Kernels with more check or variable passes than the graph occupies, which skip
the passes that it lacks, against the FP64 oracle, with and without posteriors
(rules of parity.py)."""
import pytest

import bpdc_inputs as bi
import parity
from bpdc_inputs.sampler import sample_shots
from parity import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code,kernel,opts", [
    ("bb72", 20, {}), ("bb72", 7, dict(dc_prior=1, max_iter=40)), ("bb72", 0, {}), ("bb72", 5, {}), ("bb108", 20, {}),
    ("bb144", 5, {}), ("bb72", 12, dict(variant=1)), ("bb108", 12, dict(variant=1)), ("phen", 3, dict(max_iter=60)),
    ("phen", 4, dict(max_iter=60)), ("phen", 10, dict(max_iter=60))])
def test_guarded_passes_match_the_oracle(code, kernel, opts, oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    P = bi.phenomenological_bb_problem("bb72", 6, 0.01) if code == "phen" else bi.bb_problem(code, 0.06)
    B = 400 if code == "phen" else 1500
    _, s, o = sample_shots(P, 0x2510086950, 0, B)
    opt = pkg.Options(**opts)
    g = pkg.Graph.from_problem(P, opt)
    g.set_kernel(kernel)
    out = g.decode(to_dev(s), 0, obs_true=to_dev(o), posterior=True)
    plain = g.decode(to_dev(s), 0, obs_true=to_dev(o), persistent=False)
    for k in ("corrections", "status", "logical_flips", "iterations"):
        assert bool((out[k] == plain[k]).all()), k
    oo = oracle_mod.Options(variant=opt.variant, alpha=opt.ms_scale, max_iter=opt.max_iter, dc_prior=opt.dc_prior)
    rep = parity.compare(oracle_mod, P, s, 0, oo, parity.gpu_outcome(P, out), obs=o)
    assert rep["unmatched_well"] == 0 and rep["unmatched_ill"] <= 0.02 * B, parity.summary(rep)
    assert rep["compared"] >= 0.9 * B, parity.summary(rep)
    assert rep["posterior"]["failed"] == 0 and rep["posterior"]["inf_mismatch"] == 0, rep["posterior"]
