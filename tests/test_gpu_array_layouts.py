"""Where the caller's arrays start: values of 4 bytes on any byte, in host and
device memory, read by the loads and the alignment call and written by the
result calls.  The arrays are copied bytes, so the results are equal bit for
bit to those with arrays on 16 bytes; sizes are odd, so that the copies have
remainders below 16 bytes."""
import ctypes

import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch

pytestmark = pytest.mark.gpu

OUT = dict(hits=("i4", lambda n, L: n * L), n_found=("i4", lambda n, L: n), chi2=("f4", lambda n, L: n),
           params=("f4", lambda n, L: 6 * n), cov=("f4", lambda n, L: 21 * n), keep=("u1", lambda n, L: n))


class _Array:
    """Values at `shift` bytes past a 256-byte boundary, on the device or in host memory."""

    def __init__(self, nbytes, shift, device):
        import torch
        pad = torch.zeros(nbytes + 512, dtype=torch.uint8)
        self.store = pad.cuda() if device else pad
        self.at = -self.store.data_ptr() % 256 + shift
        self.n = nbytes
        self.ptr = self.store.data_ptr() + self.at

    def put(self, a):
        import torch
        raw = np.frombuffer(np.ascontiguousarray(a).tobytes(), np.uint8).copy()
        self.store[self.at:self.at + self.n] = torch.from_numpy(raw).to(self.store.device)
        return self

    def get(self, dtype):
        return np.frombuffer(self.store[self.at:self.at + self.n].cpu().numpy().tobytes(), dtype)


def _of(a, shift, device):
    return _Array(a.nbytes, shift, device).put(a)


@pytest.mark.parametrize("device", [0, 1])
@pytest.mark.parametrize("shift", [1, 2, 3, 4])
def test_arrays_on_any_byte(shift, device):
    import torch

    from paper_1906_11744_gb300 import _lib
    b = make_batch("c1", tracks=301, misalign_sigma=0.005)
    lib = _lib.load()
    t = tracker_for(b)
    t.find_tracks()
    ref = t.get_tracks()
    t.close()

    t = tracker_for(b)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    keep = []

    def at(a):
        keep.append(_of(a, shift, device))
        return keep[-1].ptr

    off = lambda a: np.ascontiguousarray(a, np.int32).ctypes.data  # noqa: E731
    hit_off, seed_off = np.asarray(b.hit_off, np.int32), np.asarray(b.seed_off, np.int32)
    args = [at(b.x), at(b.y), at(b.z), at(b.layer)]
    sargs = [at(b.params), at(b.cov), at(b.seed_hits)]
    align = at(b.align)
    torch.cuda.synchronize()
    assert lib.kf_load_hits(t.ctx, 1, off(hit_off), *args, device, stream) == _lib.KF_OK
    assert lib.kf_load_seeds(t.ctx, 1, off(seed_off), *sargs, device, stream) == _lib.KF_OK
    assert lib.kf_set_alignment(t.ctx, align, device, stream) == _lib.KF_OK
    assert lib.kf_find_tracks(t.ctx, stream) == _lib.KF_OK
    outs = {k: _Array(f(b.n_seeds, b.det.n_layers) * np.dtype(d).itemsize, shift, device) for k, (d, f) in OUT.items()}
    assert lib.kf_get_tracks(t.ctx, *[outs[k].ptr for k in OUT], device, stream) == _lib.KF_OK
    torch.cuda.synchronize()
    for k, (d, _) in OUT.items():
        assert np.array_equal(outs[k].get(d), np.asarray(ref[k]).reshape(-1)), k
    # an index out of range is found wherever the array starts
    bad = b.layer.copy()
    bad[-1] = b.det.n_layers
    args[3] = at(bad)
    torch.cuda.synchronize()
    assert lib.kf_load_hits(t.ctx, 1, off(hit_off), *args, device, stream) == _lib.KF_ERR_ARG
    args[3] = at(b.layer)
    bad = b.seed_hits.copy()
    bad[2, -1] = b.n_hits
    sargs[2] = at(bad)
    torch.cuda.synchronize()
    assert lib.kf_load_hits(t.ctx, 1, off(hit_off), *args, device, stream) == _lib.KF_OK
    assert lib.kf_load_seeds(t.ctx, 1, off(seed_off), *sargs, device, stream) == _lib.KF_ERR_ARG
    t.close()
