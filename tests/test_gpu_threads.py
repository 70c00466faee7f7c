"""Handles of one process used from several threads at once, each thread with
its own handle and stream."""
import ctypes
import threading

import numpy as np
import pytest

import workloads as W
from gpu_common import vf  # noqa: F401

pytestmark = pytest.mark.gpu


def test_spectra_of_maps_of_different_sizes(vf):  # noqa: F811
    """The spectrograph kernel takes more or fewer warps, and shared memory, by
    the size of the map: calls of one size must not fail while other threads
    make calls of others.  The C entry point is called directly, so that the
    threads spend their time in the library."""
    v, _, torch = vf
    dev = torch.device("cuda:0")
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device=dev)  # noqa: E731
    p = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    x, c = W.spectrograph_grid()
    tf, tx = t(W.spectrograph_instrument(x, c)), t(x)
    line = v.vfisv_line(W.FE6302["lambda0_A"], W.FE6302["geff"], W.FE6302["mu"])
    cfg = v.vfisv_config_default(max_iter=0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    failed = {}

    def worker(n):
        h, s = v.vfisv_create(0), torch.cuda.Stream(dev)
        obs = v.vfisv_synth(h, t(W.quiet_and_active_params(n, n)), tf, tx, W.FE6302)
        obs = obs.reshape(n, -1).contiguous()
        w = torch.full((obs.shape[1],), 1e6, device=dev)
        ref = v.vfisv_invert(h, obs, w, tf, tx, W.FE6302, want_cov=False, config={"max_iter": 0})
        out = {k: None if r is None else torch.empty_like(r) for k, r in ref.items()}
        torch.cuda.synchronize()
        f = v.load().vfisv_invert
        args = (h.ptr, p(obs), p(w), 0, p(tf), len(tf), p(tx), len(tx), ctypes.byref(line), None,
                ctypes.byref(cfg), n, p(out["params"]), p(out["chi2"]), p(out["iters"]),
                p(out["status"]), None, ctypes.c_void_p(s.cuda_stream))

        def run():
            failed[n] = sum(1 for _ in range(5000) if f(*args) != 0)
            s.synchronize()
        return h, run, ref, out, (obs, w)  # (the arguments hold addresses only)

    jobs = [worker(n) for n in (1, 2 * sms + 1, 4 * sms + 1, 8 * sms + 1)]
    threads = [threading.Thread(target=j[1]) for j in jobs]
    for q in threads:
        q.start()
    for q in threads:
        q.join()
    assert not any(failed.values()), failed
    for h, _, ref, out, _ in jobs:
        v.vfisv_check(h)
        for k in ref:
            assert ref[k] is None or torch.equal(ref[k], out[k]), k
        h.close()
