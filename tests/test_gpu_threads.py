"""Host threads on streams of their own, launching the same kernels with different amounts of shared memory: none
lowers the limit another thread's launch needs, and results equal those of one thread."""
import threading

import pytest
import torch

import paper_2508_10307_gb300 as H
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
def test_threads_with_different_windows(batch):
    x = torch.from_numpy(synth.add_gaussian(synth.clean_image(64, 72, 3, 3), 20.0, 3)).cuda()
    params = [dict(stride=3, window=w, K=8, tile=t) for w, t in ((7, 1), (24, 8), (12, 3), (30, 6))]

    def call(p):
        return H.denoise_batch([x, x], [20.0] * 2, p)[1] if batch else H.denoise(x, 20.0, p)

    want = [call(p) for p in params]
    torch.cuda.synchronize()
    failed = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(150):
                    got = call(params[k])
                torch.cuda.current_stream().synchronize()
                assert torch.equal(got, want[k])
        except Exception as e:
            failed.append((k, e))

    th = [threading.Thread(target=work, args=(k,)) for k in range(len(params))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not failed, failed
