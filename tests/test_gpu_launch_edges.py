"""Launch edges of the kernels with an instance of their own for launches of one
batch, and lists of as many batches as travel with a launch or need copied
descriptors, are split over launches, or hold empty batches; each equal to one
large decode."""
import pytest

import bpdc_inputs as bi

pytestmark = pytest.mark.gpu
KEYS = ("corrections", "status", "logical_flips", "iterations")
# code -> problem, options, kernel
CODES = {"bb72": (lambda: bi.bb_problem("bb72", 0.06), {}, 19),
         "bb108": (lambda: bi.bb_problem("bb108", 0.06), {}, 21),
         "bb144": (lambda: bi.bb_problem("bb144", 0.06), {}, 20),
         "surface5": (lambda: bi.surface_problem(5, 0.06), dict(variant=1, max_iter=25, dc_prior=1), 11),
         "bb72_product_sum": (lambda: bi.bb_problem("bb72", 0.06), dict(variant=1), 12),
         "phenomenological": (lambda: bi.phenomenological_bb_problem("bb72", 6, 0.008), dict(max_iter=30), 3)}


@pytest.fixture(scope="module", params=sorted(CODES))
def case(request):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    make, opts, kernel = CODES[request.param]
    g = pkg.Graph.from_problem(make(), pkg.Options(**opts))
    assert g.info["kernel_id"] == kernel
    syn, obs, _ = g.sample(6000, 3, 0)
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    ref = g.decode(syn, 0, obs_true=obs, counters=cnt)
    return torch, pkg, g, syn, obs, ref, cnt


@pytest.mark.parametrize("B", [1, 7, 152, 153, 1216, 1217, 4865])
@pytest.mark.parametrize("persistent", [True, False])
def test_one_batch(case, B, persistent):
    torch, pkg, g, syn, obs, ref, _ = case
    for first in (0, 6000 - B):
        out = g.decode(syn[first:first + B].contiguous(), first, persistent=persistent)
        assert all(torch.equal(out[k], ref[k][first:first + B]) for k in KEYS)


@pytest.mark.parametrize("n", [1, 2, 4, 5, 16, 17, 32, 33])
@pytest.mark.parametrize("empty", [False, True])
@pytest.mark.parametrize("noalloc", [True, False])
def test_lists(case, n, empty, noalloc):
    torch, pkg, g, syn, obs, ref, cnt = case
    size = [1 + (37 * i + 11) % 180 for i in range(n)]   # none empty
    if empty:
        size = [b for s in size for b in (s, 0)]
    if noalloc and len(size) > 16:
        pytest.skip("at most 16 batches")
    rest = 6000 - sum(size)
    for _ in range(2):   # launch after launch on the same counters
        items, at = [], 0
        counters = torch.zeros(4, dtype=torch.int64, device="cuda")
        for b in size:
            items.append(dict(graph=g, syndromes=syn[at:at + b].contiguous(), obs_true=obs[at:at + b].contiguous(),
                              shot_offset=at, out=g.alloc_outputs(b), counters=counters))
            at += b
        (pkg.decode_multi_noalloc if noalloc else pkg.decode_multi)(items)
        g.decode(syn[at:].contiguous(), at, obs_true=obs[at:].contiguous(), counters=counters)
        at = 0
        for it, b in zip(items, size):
            assert all(torch.equal(it["out"][k], ref[k][at:at + b]) for k in KEYS)
            at += b
        assert rest > 0 and torch.equal(counters, cnt)
