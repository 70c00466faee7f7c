"""Handles of one process used from several threads at once, each thread with
its own handle and stream.  A kernel's limit of shared memory is one for all of
them, while the bytes a call needs go by its map and its grid.  The C entry
point is called directly, so that the threads spend their time in the library."""
import ctypes
import threading

import numpy as np
import pytest

import workloads as W
from gpu_common import vf  # noqa: F401

pytestmark = pytest.mark.gpu


def _together(v, torch, jobs, reps=5000):
    """jobs: (handle, T, x, line, pixels); every call must succeed and every
    thread's last outputs be those of a call by itself."""
    dev = torch.device("cuda:0")
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device=dev)  # noqa: E731
    p = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    cfg = v.vfisv_config_default(max_iter=0)
    f = v.load().vfisv_invert
    failed, work = {}, []
    for i, (h, T, x, ln, n) in enumerate(jobs):
        tf, tx, s = t(T), t(x), torch.cuda.Stream(dev)
        obs = v.vfisv_synth(h, t(W.quiet_and_active_params(n, n)), tf, tx, ln)
        obs = obs.reshape(n, -1).contiguous()
        w = torch.full((obs.shape[1],), 1e6, device=dev)
        ref = v.vfisv_invert(h, obs, w, tf, tx, ln, want_cov=False, config={"max_iter": 0})
        out = {k: None if r is None else torch.empty_like(r) for k, r in ref.items()}
        line = v.vfisv_line(ln["lambda0_A"], ln["geff"], ln["mu"])
        args = (h.ptr, p(obs), p(w), 0, p(tf), len(tf), p(tx), len(tx), ctypes.byref(line), None,
                ctypes.byref(cfg), n, p(out["params"]), p(out["chi2"]), p(out["iters"]),
                p(out["status"]), None, ctypes.c_void_p(s.cuda_stream))

        def run(i=i, args=args, s=s):
            failed[i] = sum(1 for _ in range(reps) if f(*args) != 0)
            s.synchronize()
        # (the arguments hold addresses only: what they point to is kept here)
        work.append((threading.Thread(target=run), h, ref, out, (tf, tx, obs, w, line)))
    torch.cuda.synchronize()
    for q in work:
        q[0].start()
    for q in work:
        q[0].join()
    assert not any(failed.values()), failed
    for _, h, ref, out, _ in work:
        v.vfisv_check(h)
        for k in ref:
            assert ref[k] is None or torch.equal(ref[k], out[k]), k
        h.close()


def test_spectra_of_maps_of_different_sizes(vf):  # noqa: F811
    """The spectrograph kernel takes more or fewer warps by the size of the map."""
    v, _, torch = vf
    x, c = W.spectrograph_grid()
    T = W.spectrograph_instrument(x, c)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _together(v, torch, [(v.vfisv_create(0), T, x, W.FE6302, n)
                         for n in (1, 2 * sms + 1, 4 * sms + 1, 8 * sms + 1)])


@pytest.mark.parametrize("shapes", [(384, 128, 384, 128), (0, 0, 0, 0)])
def test_grids_of_different_lengths(vf, shapes):  # noqa: F811
    """A longer grid has a larger filter table, and the choice of a kernel asks
    about others than the one it takes."""
    v, _, torch = vf
    jobs = []
    for block, nlam, n in zip(shapes, (75, 600, 149, 2000), (300, 200, 2000, 100)):
        h = v.vfisv_create(0)
        v.vfisv_set_launch_shape(h, block, 1)
        x = np.linspace(-740.0, 740.0, nlam)
        jobs.append((h, W.hmi_filters(x), x, W.FE6173, n))
    _together(v, torch, jobs)
