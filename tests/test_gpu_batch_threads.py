"""Batch calls of several host threads on one stream (every Python thread's default one): the lanes and their
workspaces belong to the stream, so the calls take turns. Results equal those of the thread's images alone."""
import threading

import pytest
import torch

import paper_2508_10307_gb300 as H
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


def test_threads_share_a_stream():
    prm = dict(stride=3, window=9, K=8)
    sizes = [[(40, 64), (117, 122), (60, 33)], [(96, 200), (33, 33)], [(64, 64)] * 5, [(150, 40)]]
    sets = [[torch.from_numpy(synth.add_gaussian(synth.clean_image(h, w, 3, 7 * k + i), 20.0, i)).cuda()
             for i, (h, w) in enumerate(hw)] for k, hw in enumerate(sizes)]
    want = [H.denoise_batch(xs, [20.0] * len(xs), prm) for xs in sets]
    torch.cuda.synchronize()
    H.load_library().htsvd_release_workspace()       # (the workspaces grow while the threads call)
    bad = []

    def work(k):
        for _ in range(20):
            got = H.denoise_batch(sets[k], [20.0] * len(sets[k]), prm)
            torch.cuda.current_stream().synchronize()
            if not all(torch.equal(a, b) for a, b in zip(got, want[k])):
                bad.append(k)

    th = [threading.Thread(target=work, args=(k,)) for k in range(len(sets))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad
