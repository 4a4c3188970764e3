"""Lists that mix BB[[108,8,10]] (variant 21) with BB[[144,12,12]] (variant 20): one
decode kernel where the former's shots are few, two where they are many, and the
results of each batch alone either way."""
import ctypes

import pytest

import bpdc_inputs as bi

pytestmark = pytest.mark.gpu


def _kernels(torch, pkg, items):
    """Kernel launches of an allocation-free call: the nodes of its graph (a setup
    and a decode kernel for each launch)."""
    pkg.decode_multi_noalloc(items)
    torch.cuda.synchronize()
    try:
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        cudart = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    except (TypeError, OSError):
        return None
    stream = torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        pkg.decode_multi_noalloc(items, stream)
    n = ctypes.c_size_t()
    assert cudart.cudaGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    graph.instantiate()
    graph.replay()
    torch.cuda.synchronize()
    return n.value


@pytest.mark.parametrize("p,small,other,posterior,launches", [
    (0.05, 1, 1, False, 1), (0.05, 64, 700, True, 1), (0.05, 20000, 1000, False, 1), (0.02, 60000, 10, False, 1),
    (0.05, 40000, 1000, False, 2), (0.08, 15000, 64, False, 2), (0.05, 300, 0, False, 1), (0.05, 0, 300, False, 1)])
def test_mixed_lists(p, small, other, posterior, launches):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    items, ref = [], []
    for code, shots in (("bb108", small), ("bb144", other), ("bb108", small // 7)):
        g = pkg.Graph.from_problem(bi.bb_problem(code, p))
        assert g.info["kernel_id"] == (21 if code == "bb108" else 20)
        syn, obs, _ = g.sample(shots, 7, 100)
        cnt = [torch.zeros(4, dtype=torch.int64, device="cuda") for _ in range(2)]
        out = g.alloc_outputs(shots, posterior=posterior)
        ref.append((g.decode(syn, 100, obs_true=obs, counters=cnt[1], posterior=posterior), cnt[1]))
        items.append(dict(graph=g, syndromes=syn, obs_true=obs, shot_offset=100, out=out, counters=cnt[0]))

    def check():
        torch.cuda.synchronize()
        for it, (r, c) in zip(items, ref):
            for k, v in it["out"].items():
                assert torch.equal(v, r[k]), k
                v.zero_()
            assert torch.equal(it["counters"], c)
            it["counters"].zero_()

    pkg.decode_multi(items)
    check()
    pkg.decode_multi_noalloc(items)
    check()
    n = _kernels(torch, pkg, items)
    assert n is None or n == 2 * launches
