"""Two contexts with different checkpoint strides in two host threads: the
adjoint kernels' shared-memory limit belongs to the kernel and not to a
context, so neither thread may lower it under the other's launch."""
import threading

import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch
from synth.events import true_hit_lists

pytestmark = pytest.mark.gpu


def test_adjoints_of_two_strides_at_once():
    import torch

    from paper_1906_11744_gb300 import KF_FIT_GIVEN
    b = make_batch("c3", tracks=100)
    lists, nh = true_hit_lists(b, 0, b.det.n_layers)
    lists, nh = lists[b.seed_sim], nh[b.seed_sim]
    dev = torch.device("cuda:0")
    errors, grads, start = [], {}, threading.Barrier(2)

    def work(stride):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                t = tracker_for(b, device=dev, ckpt_stride=stride)
                t.fit_tracks(KF_FIT_GIVEN, torch.from_numpy(lists).to(dev), torch.from_numpy(nh).to(dev), stream)
                g = [torch.zeros(s, dtype=torch.float32, device=dev) for s in ((b.det.n_layers, 2), (b.n_hits, 3))]
                start.wait()
                for _ in range(1500):
                    t.fit_adjoint(g[0], g[1], None, stream)
                stream.synchronize()
                grads[stride] = g[1].cpu().numpy()
                t.close()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
            start.abort()

    threads = [threading.Thread(target=work, args=(s,)) for s in (1, 8)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    assert np.abs(grads[1] - grads[8]).max() < 1e-3 * np.abs(grads[1]).max()
