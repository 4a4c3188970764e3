"""The work counter of the allocation-free decode is set at the start of every
call: calls that overlapped (which the header forbids: they share the counter and
spoil each other's results, within their own buffers) leave no trace in the next
call, nor in the next replay of a captured one."""
import pytest

import bpdc_inputs as bi

pytestmark = pytest.mark.gpu
KEYS = ("corrections", "status", "logical_flips", "iterations")


@pytest.mark.parametrize("n", [1, 5])
def test_a_call_after_overlapping_calls_is_whole(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_08695_gb300 as pkg
    big = pkg.Graph.from_problem(bi.hgp_problem(0.06))
    small = pkg.Graph.from_problem(bi.bb_problem("bb72", 0.06))

    def items(g, shots, batches):
        syn, _, _ = g.sample(shots, 3, 0)
        return [dict(graph=g, syndromes=syn, shot_offset=0, out=g.alloc_outputs(shots)) for _ in range(batches)]

    long_call, short_call, call = items(big, 6000, 1), items(small, 3000, 1), items(small, 3000, n)
    ref = small.decode(call[0]["syndromes"], 0)
    pkg.decode_multi_noalloc(call)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        pkg.decode_multi_noalloc(call, stream)
    for run in (lambda: pkg.decode_multi_noalloc(call), graph.replay):
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        pkg.decode_multi_noalloc(long_call, a)
        for _ in range(3):
            pkg.decode_multi_noalloc(short_call, b)
        torch.cuda.synchronize()
        for it in call:
            for k in KEYS:
                it["out"][k].fill_(-1 if k != "status" else 255)
        run()
        torch.cuda.synchronize()
        assert all(torch.equal(it["out"][k], ref[k]) for it in call for k in KEYS)
