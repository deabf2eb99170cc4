"""Handles of different sizes on different host threads: one thread's launches do not depend on another's."""
import threading

import numpy as np
import pytest

from gpu_util import System, ensure_built, params_for, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shapes", [
    ("FCM_FP32", [((8, 8, 256), 8, 0), ((8, 8, 80), 8, 0)]),      # columns in z of 256 and 80 points
    ("FCM_FP64", [((8, 8, 128), 8, 0), ((8, 8, 54), 8, 0)]),
    ("FCM_FP32", [((24, 24, 24), 11, 0), ((24, 24, 24), 9, 0)]),  # supports that share a compiled variant
    ("FCM_FP32", [((24, 24, 24), 11, 2), ((24, 24, 24), 9, 2)]),  # the same in the shared-atomics spread
])
def test_threads_with_handles_of_their_own(precision, shapes):
    """Each thread applies its handle a thousand times; every status is FCM_OK and every result agrees with the one
    computed before the threads started to the rounding of sums whose order is not fixed (1e-5 in FP32, 1e-12 in FP64;
    a launch that did not run leaves the result of other loads)."""
    torch = torch_cuda()
    fcm = ensure_built()
    prec = getattr(fcm, precision)
    dt, bar = (torch.float32, 1e-5) if prec == fcm.FCM_FP32 else (torch.float64, 1e-12)
    jobs = []
    for k, (M, M_G, kernel) in enumerate(shapes):
        s = System(30, tuple(1.1 * m for m in M), M, 0.9, min(M_G, min(M)), 3.0, 60 + k)
        p = params_for(fcm, s, prec)
        p.spread_kernel = kernel
        arrays = [torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda:0") for a in (s.Y, s.F, s.T)]
        jobs.append((fcm.Handle(p), torch.cuda.Stream(), arrays, s.n))
    torch.cuda.synchronize()   # the streams below do not wait for the copies above by themselves
    ref = [fcm.apply_tensors(h, *a, stream=st.cuda_stream) for h, st, a, _ in jobs]
    torch.cuda.synchronize()
    loads = [(-F, -T) for _, _, (_, F, T), _ in jobs]
    torch.cuda.synchronize()
    errors, got = [], [None] * len(jobs)

    def work(k):
        h, st, (pos, F, T), n = jobs[k]
        U, W = torch.zeros_like(F), torch.zeros_like(F)
        try:
            for it in range(1000):   # an even call's loads have the other sign, so a call that did nothing shows
                h.apply(n, pos, *((F, T) if it % 2 else loads[k]), U, W, st.cuda_stream)
                if it % 50 == 49:
                    st.synchronize()
            got[k] = (U, W)
        except fcm.FcmError as e:
            errors.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for h, _, _, _ in jobs:
        h.close()
    assert not errors, errors[:3]
    for k in range(len(jobs)):
        for a, b in zip(got[k], ref[k]):
            assert rel_l2(a.double().cpu().numpy(), b.double().cpu().numpy()) < bar
