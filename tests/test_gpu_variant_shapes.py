"""The variant of the BB[[108,8,10]] shape (two check and four variable passes of
a warp) at the edges of what it takes: it is the automatic choice where the
three- and five-pass variant was, every variant decodes alike, and an
allocation-free launch still mixes its graphs with that variant's."""
import numpy as np
import pytest
import scipy.sparse as sp

import bpdc_inputs as bi
from bpdc_inputs.codes import Problem, _csr

pytestmark = pytest.mark.gpu


def _regular(M):
    """M checks of weight 6 on 2M columns of weight 3 (two circulant blocks)."""
    j = np.arange(M)
    rows = np.concatenate([(j + s) % M for s in (0, 1, 5)] + [(j + s) % M for s in (0, 2, 9)])
    cols = np.concatenate([j, j, j, M + j, M + j, M + j])
    H = _csr(sp.csr_matrix((np.ones(6 * M, np.uint8), (rows, cols)), shape=(M, 2 * M)))
    rng = np.random.default_rng(M)
    D = _csr(sp.csr_matrix((np.ones(6 * M, np.uint8), (rows, (cols + 3) % (2 * M))), shape=(M, 2 * M)))
    return Problem(f"regular{M}", H, D, _csr(rng.random((5, 2 * M)) < 0.3), np.full(2 * M, 0.06))


@pytest.mark.parametrize("M,auto", [(49, 21), (54, 21), (63, 21), (64, 21), (65, 20)])
def test_two_pass_shape(M, auto):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    g = pkg.Graph.from_problem(_regular(M))
    assert g.info["kernel_id"] == auto
    syn, obs, _ = g.sample(3000, 5, 0)
    ref = g.decode(syn, 0, obs_true=obs)
    soft = g.decode(syn, 0, obs_true=obs, posterior=True)
    for k in g.kernels():
        g.set_kernel(k)
        out = g.decode(syn, 0, obs_true=obs)
        assert all(torch.equal(out[x], ref[x]) for x in ref), k
    assert all(torch.equal(soft[x], ref[x]) for x in ref)
    g.set_kernel(auto)
    other = pkg.Graph.from_problem(bi.bb_problem("bb144", 0.05))
    s2, o2, _ = other.sample(700, 5, 0)
    items = [dict(graph=h, syndromes=s, obs_true=o, shot_offset=0, out=h.alloc_outputs(s.shape[0]))
             for h, s, o in ((other, s2, o2), (g, syn, obs), (other, s2, o2))]
    pkg.decode_multi_noalloc(items)
    r2 = other.decode(s2, 0, obs_true=o2)
    for it, r in zip(items, (r2, ref, r2)):
        assert all(torch.equal(it["out"][x], r[x]) for x in r)


@pytest.mark.parametrize("code,kept,stored", [("bb72", (19, 17, 20, 7), 5), ("regular54", (21, 20), 3), ("bb144", (20, 0), 10)])
@pytest.mark.parametrize("max_iter,dc", [(0, 1), (1, 0), (20, 1)])
def test_kept_posteriors(code, kept, stored, max_iter, dc):
    """Posteriors kept in registers until the run ends equal those stored at every
    iteration: converged, failed, after a cut, for a zero syndrome and on a given
    cut set."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    P = _regular(54) if code == "regular54" else bi.bb_problem(code, 0.06)
    g = pkg.Graph.from_problem(P, pkg.Options(max_iter=max_iter, dc_enable=dc, dc_prior=dc))
    syn, _, _ = g.sample(500, 5, 0)
    syn[7] = 0
    cut = g.cut_select(torch.randn((500, g.N), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda"))
    g.set_kernel(stored)
    ref = [g.decode(syn, 0, posterior=True), g.decode(syn, 0, posterior=True, cut_in=cut, persistent=False)]
    for k in kept:
        g.set_kernel(k)
        out = [g.decode(syn, 0, posterior=True), g.decode(syn, 0, posterior=True, cut_in=cut, persistent=False)]
        for a, b in zip(out, ref):
            assert all(torch.equal(a[x], b[x]) for x in b), k
