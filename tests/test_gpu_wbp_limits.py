"""The edge limit of weighted BP: a larger graph is UNSUPPORTED, by name and for
both calls, the largest runs, and neither depends on the checkpoint interval."""
import numpy as np
import pytest
import scipy.sparse as sp

from bpdc_inputs.codes import Problem, _csr

pytestmark = pytest.mark.gpu


def _graph(pkg, M):
    """M checks of weight 8 on 4M columns of weight 2: 8M edges."""
    j = np.arange(4 * M)
    rows, cols = np.concatenate([j % M, (j + 1 + j // M) % M]), np.concatenate([j, j])
    H = _csr(sp.csr_matrix((np.ones(8 * M, np.uint8), (rows, cols)), shape=(M, 4 * M)))
    none = sp.csr_matrix((0, 4 * M), dtype=np.uint8)
    return pkg.Graph.from_problem(Problem(f"edges{8 * M}", H, none, none, np.full(4 * M, 0.02)))


@pytest.mark.parametrize("M,fits", [(380, True), (454, True), (455, False), (600, False)])
def test_edge_limit(M, fits):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    from paper_2510_08695_gb300 import _bpdc
    g = _graph(pkg, M)
    B, T = 3, 10
    syn, _, _ = g.sample(B, 7, 0)
    gen = torch.Generator(device="cuda").manual_seed(M)
    W = 1 + 0.1 * torch.randn((2, T, g.E), generator=gen, device="cuda")
    up = torch.randn((B, T, g.N), generator=gen, device="cuda")
    outs = []
    for k in (1, 5, T):
        ws = _bpdc.wbp_workspace(g, B, T, k)
        calls = (lambda: _bpdc.wbp_forward(g, syn, W, T, 20.0, k, ws),
                 lambda: _bpdc.decode_backward(g, syn, W, T, 20.0, k, up, ws))
        if fits:
            outs.append([c() for c in calls])
            continue
        for c in calls:
            with pytest.raises(pkg.BpdcError) as err:
                c()
            assert err.value.code == _bpdc.ERR_UNSUPPORTED and "3632 edges" in str(err.value)
    for o in outs[1:]:
        assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])
    assert all(bool(x.isfinite().all()) for o in outs for x in o)
