"""Device evaluations on a stream that is capturing: one that the call before has prepared is recorded and
replays with the bits of a direct call; one that would need set-up (tables, buffers, another key) is
refused, and the context works afterwards."""
import numpy as np
import pytest

import musr_inputs as mi
import oracle
from test_gpu_parity import _check_fp64, _check_split

pytestmark = pytest.mark.gpu


def test_calls_under_capture(musr_lib):
    import torch

    from paper_1509_07685_gb300 import binding as B
    p = mi.cfg2(nhist=8, nbins=3001, bin_width_ns=4.0, seed=83)
    X = mi.jitter(p.truth, 2, seed=2, lo=0.98, hi=1.02)
    stream = torch.cuda.Stream()
    x = torch.empty((2, p.nparams), dtype=torch.float64, device="cuda")
    out = torch.full((2, 1 + p.nparams), float("nan"), dtype=torch.float64, device="cuda")
    for prec, check in ((B.MUSR_SPLIT, _check_split), (B.MUSR_FP64, _check_fp64)):
        x.copy_(torch.tensor(X))
        torch.cuda.synchronize()
        with B.Context(p, cuda_stream=stream.cuda_stream) as ctx:
            call = lambda n, row: B.musr_eval_device(ctx.ctx, x[row:].data_ptr(), n, 1, prec, True, out[row:].data_ptr())

            def refused(n):
                with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=stream, capture_error_mode="relaxed"):
                    with pytest.raises(B.MusrError) as e:
                        call(n, 0)
                return e.value.status == B.MUSR_ESTATE and "capturing" in str(e.value)

            assert refused(1)  # nothing is set up yet
            call(1, 0)
            torch.cuda.synchronize()
            check(out[0, 0].item(), out[0, 1:].cpu().numpy(), oracle.cost(p, X[0], 1))
            assert refused(2)  # another key
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream, capture_error_mode="relaxed"):
                call(1, 1)  # other buffers, the same key
            for params in X:  # replays follow the buffers' contents; a direct call gives the same bits
                x.copy_(torch.tensor(np.stack([params, params])))
                g.replay()
                torch.cuda.synchronize()
                call(1, 0)
                torch.cuda.synchronize()
                assert torch.equal(out[0], out[1])
                check(out[1, 0].item(), out[1, 1:].cpu().numpy(), oracle.cost(p, params, 1))
