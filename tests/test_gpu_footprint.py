"""Device memory of an exploration job as the request loop counts it
(rid_submit refuses a job larger than the server's budget).  The ensemble's
scratch is counted in whole tiles of the walkers that the call has: 128 walkers
for the tensor-core ensembles (saved tanh, residual stream, 32 partial sums each),
32 walkers of saved tanh at most for FP32."""
import re

import numpy as np
import pytest

from paper_2408_14070_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2408_14070_gb300 import build, rid
    build.build()
    return rid


def _needed(R, sysobj, x0, steps):
    with R.Server(1 << 20) as srv:            # the smallest budget
        with pytest.raises(R.RidError) as e:
            srv.cancel(srv.submit_explore(sysobj, x0, steps, x_out=np.zeros_like(x0)))
    return int(re.search(r"needs (\d+) bytes", str(e.value))[1])


def _bound(sp, ens, W, prec, resnet, steps):
    N, C, M, L, H = sp.n_beads, sp.n_cv, ens.n_models, ens.n_layers, (ens.width + 31) // 32 * 32
    b = 64 * W * N + W * C * 76 + 16 * W + 24 * W * N + M * W * C * 4 + M * W * 4
    if prec == "fp32":
        b += M * L * H * 32 * ((W + 31) // 32) * 4
    else:
        b += M * ((W + 127) // 128) * 128 * (H * (2 * L + (4 if resnet else 0)) + 32 * 4)
    of = sp.output_freq
    chunk = max(W * (steps // of) * (C + 1) * 4, W * N * 24)      # one replayed chunk of outputs at most
    return b + (chunk + 255) // 256 * 256


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("W,H,resnet", [(12, 300, True), (128, 256, False), (129, 256, False), (300, 512, False),
                                        (640, 64, True)])
def test_tensor_core_scratch_is_counted_in_tiles_of_128_walkers(R, prec, W, H, resnet):
    sp = I.make_system(30, 6, 3, output_freq=10)
    ens = I.make_ensemble(8, 12, 2, H, 3, resnet=resnet)
    x0 = I.make_chains(W, sp, 3)
    with R.System(sp) as s:
        s.set_ensemble(ens, precision={"bf16": R.RID_PREC_BF16, "fp8": R.RID_PREC_FP8}[prec])
        assert _needed(R, s, x0, 20) <= _bound(sp, ens, W, prec, resnet, 20)


@pytest.mark.parametrize("W,H,resnet", [(12, 300, True), (33, 256, False), (1000, 128, False), (1999, 256, True)])
def test_fp32_scratch_is_counted_for_the_walkers_of_the_call(R, W, H, resnet):
    sp = I.make_system(30, 6, 3, output_freq=10)
    ens = I.make_ensemble(16, 12, 4, H, 3, resnet=resnet)
    x0 = I.make_chains(W, sp, 3)
    with R.System(sp) as s:
        s.set_ensemble(ens, precision=R.RID_PREC_FP32)
        assert _needed(R, s, x0, 20) <= _bound(sp, ens, W, "fp32", resnet, 20)
