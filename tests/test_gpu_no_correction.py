"""FCM_STAGE_PAIR alone on a handle whose correction is identically zero (Sigma = sigma, Sigma_D = sigma_D): zeros, in
both precisions and in a batch, and the check of the positions as in any other call."""
import pytest

from gpu_util import SIGMA, SIGMA_D, System, ensure_built, params_for, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["FCM_FP32", "FCM_FP64"])
@pytest.mark.parametrize("systems", [1, 3])
def test_pair_stage_without_correction(precision, systems):
    torch = torch_cuda()
    fcm = ensure_built()
    prec = getattr(fcm, precision)
    dt = torch.float32 if prec == fcm.FCM_FP32 else torch.float64
    s = System(90, 24.0, 32, SIGMA, 8, 0.0, 4, Sigma_D=SIGMA_D)
    to = lambda a: torch.as_tensor(a, dtype=dt, device="cuda:0")
    pos, F, T = to(s.Y), to(s.F), to(s.T)
    U, W = torch.full_like(F, 7.0), torch.full_like(F, 7.0)
    stream = torch.cuda.current_stream().cuda_stream
    with fcm.Handle(params_for(fcm, s, prec), 0, systems) as h:
        def call():
            if systems == 1:
                h.apply_stages(s.n, pos, F, T, U, W, fcm.STAGE_PAIR, stream)
            else:
                h.batch_apply([0, 40, 40, s.n], pos, F, T, U, W, stream, fcm.STAGE_PAIR)

        call()
        assert h.check(stream) == 0
        assert not U.any() and not W.any()
        pos[17, 1] = float("nan")
        call()
        assert h.check(stream) == fcm.STATUS_NONFINITE
