"""Launches at the edges of their shapes: shots fewer than, as many as and just
above the SMs and the resident groups, and batch lists that just fit a launch's
own parameters or need the copied descriptors; each equal to one large decode."""
import pytest

import bpdc_inputs as bi

pytestmark = pytest.mark.gpu
KEYS = ("corrections", "status", "logical_flips", "iterations")


@pytest.fixture(scope="module")
def case():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    g = pkg.Graph.from_problem(bi.bb_problem("bb72", 0.06))
    syn, obs, _ = g.sample(12000, 3, 0)
    ref = g.decode(syn, 0, obs_true=obs)
    return torch, pkg, g, syn, ref


@pytest.mark.parametrize("B", [1, 2, 8, 151, 152, 153, 304, 305, 1215, 1216, 1217, 4864, 4865, 9000])
@pytest.mark.parametrize("persistent", [True, False])
def test_small_batches(case, B, persistent):
    torch, pkg, g, syn, ref = case
    for first in (0, 12000 - B):
        out = g.decode(syn[first:first + B].contiguous(), first, persistent=persistent)
        assert all(torch.equal(out[k], ref[k][first:first + B]) for k in KEYS)


@pytest.mark.parametrize("n", [1, 4, 5, 16, 32, 33, 70])
@pytest.mark.parametrize("noalloc", [True, False])
def test_batch_lists(case, n, noalloc):
    torch, pkg, g, syn, ref = case
    if noalloc and n > 16:
        pytest.skip("at most 16 batches")
    size = [(7 * i) % 90 for i in range(n)]   # empty and uneven batches
    for _ in range(3):                        # launch after launch on the same counters
        items, at = [], 0
        for b in size:
            items.append(dict(graph=g, syndromes=syn[at:at + b].contiguous(), shot_offset=at, out=g.alloc_outputs(b)))
            at += b
        (pkg.decode_multi_noalloc if noalloc else pkg.decode_multi)(items)
        at = 0
        for it, b in zip(items, size):
            assert all(torch.equal(it["out"][k], ref[k][at:at + b]) for k in KEYS)
            at += b
