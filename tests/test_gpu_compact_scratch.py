"""The scratch of dtb_spike_compact comes from a pool of the library's: calls on
several streams at once, after a synchronisation and inside a captured graph
give the ids of the bits each was handed."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bits(n, seed):
    import torch

    fired = np.random.default_rng(seed).random(n) < 0.01
    pad = np.zeros(-(-n // 1024) * 1024, bool)
    pad[:n] = fired
    return torch.from_numpy(np.packbits(pad, bitorder="little").view(np.int32)).cuda(), np.flatnonzero(fired)


def test_compaction_on_streams_and_in_a_graph():
    import torch

    from paper_2308_01241_gb300 import dtb

    sizes = [1000, 1025, 65536 * 3 + 7, 2_000_001]
    sets = [_bits(n, n) for n in sizes]
    out = [(torch.full((n,), -1, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"))
           for n in sizes]

    def check():
        torch.cuda.synchronize()
        for (bits, want), (ids, cnt) in zip(sets, out):
            k = int(cnt.item())
            np.testing.assert_array_equal(ids[:k].cpu().numpy(), want)
            ids.fill_(-1)
            cnt.zero_()
        torch.cuda.synchronize()

    # inside a graph, each call's scratch a part of it
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        for n, (bits, _), (ids, cnt) in zip(sizes, sets, out):
            dtb.dtb_spike_compact(bits, n, ids, cnt, side.cuda_stream)
    for _ in range(2):
        graph.replay()
        check()

    def work(q):
        st = torch.cuda.Stream()
        for _ in range(50):
            dtb.dtb_spike_compact(sets[q][0], sizes[q], out[q][0], out[q][1], st.cuda_stream)
        st.synchronize()

    threads = [threading.Thread(target=work, args=(q,)) for q in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    check()
