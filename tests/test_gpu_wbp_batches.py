"""Weighted BP does not depend on how shots share the GPU: posteriors of a batch
equal those of its shots decoded alone bit for bit, and the gradient of a batch
is the sum of its parts' gradients.  Batches at the edges of the launch: a shot
alone, one block, blocks in several rounds, uneven last blocks, teams of 256 and
of 64 threads; narrow and general row / column widths."""
import numpy as np
import pytest
import scipy.sparse as sp

import bpdc_inputs as bi
from bpdc_inputs.codes import Problem, _csr

pytestmark = pytest.mark.gpu


def _wide_graph():
    """60 checks of weight 10, 120 columns of weight 5 (beyond the narrow widths)."""
    rows = np.concatenate([(np.arange(120) * 7 + s) % 60 for s in (0, 1, 5, 13, 29)])
    H = _csr(sp.csr_matrix((np.ones(600, np.uint8), (rows, np.tile(np.arange(120), 5))), shape=(60, 120)))
    return Problem("wide", H, sp.csr_matrix((0, 120), dtype=np.uint8), sp.csr_matrix((0, 120), dtype=np.uint8),
                   np.full(120, 0.03))


GRAPHS = {"bb72": lambda: bi.bb_problem("bb72", 0.06), "surface5": lambda: bi.surface_problem(5, 0.05),
          "wide": _wide_graph}


@pytest.mark.parametrize("code,T,B,part", [("bb72", 6, 3, 1), ("bb72", 1, 4, 1), ("bb72", 6, 5, 1), ("bb72", 6, 33, 1),
                                           ("surface5", 4, 9, 1), ("wide", 5, 13, 1), ("bb72", 4, 1217, 100),
                                           ("bb72", 3, 1100, 100), ("wide", 3, 2500, 250)])
def test_batch_is_the_sum_of_its_parts(code, T, B, part):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    from paper_2510_08695_gb300 import wbp
    P = GRAPHS[code]()
    g = pkg.Graph.from_problem(P, pkg.Options(variant=0 if code == "wide" else 1, max_iter=T))
    syn, _, _ = g.sample(B, 11, 0)
    gen = torch.Generator(device="cuda").manual_seed(B)
    W = 1 + 0.1 * torch.randn((2, T, g.E), generator=gen, device="cuda")
    up = torch.randn((B, T, g.N), generator=gen, device="cuda")

    def step(a, b):
        w = W.clone().requires_grad_(True)
        post = wbp.weighted_bp(w, g, syn[a:b].contiguous(), 20.0, 1)
        post.backward(up[a:b].contiguous())
        return post.detach(), w.grad.double()

    post, grad = step(0, B)
    total, size = torch.zeros_like(grad), grad.abs()
    for a in range(0, B, part):
        p, gr = step(a, min(B, a + part))
        assert torch.equal(p, post[a:a + part])
        total += gr
        size += gr.abs()
    # every part and the total are sums rounded once to 24 bits
    assert ((grad - total).abs() <= size * 2.0 ** -24 + 1e-37).all()
