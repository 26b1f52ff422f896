"""Evaluations from several host threads, each with its own context and stream, in
shapes that share a kernel and differ in its shared memory."""
import threading

import numpy as np
import pytest

from paper_2510_25938_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


@pytest.mark.parametrize("f32", [True, False])
def test_threads_with_different_shared_memory(lj, f32):
    dt = torch.float32 if f32 else torch.float64
    prec = lj.LJ_PREC_FP32 if f32 else lj.LJ_PREC_FP64
    # one kernel each in FP32 and FP64 (groups of four): 53 and 107 KB, 90 and 102 KB
    shapes = [(500, 700), (1024, 160)] if f32 else [(800, 90), (1024, 40)]
    inputs, want = [], []
    ctx = lj.Ctx(0)
    for n, c in shapes:
        x = torch.as_tensor(I.fcc_fragments(c, n, 0.05, n).reshape(-1), device="cuda").to(dt)
        e = torch.empty(c, dtype=torch.float64, device="cuda")
        lj.lj_energy_grad_batched(ctx, x, e, None, n_cand=c, uniform_n=n, prec=prec)
        inputs.append(x)
        want.append(e.cpu().numpy())
    ctx.close()
    errors = []

    def work(k):
        try:
            n, c = shapes[k]
            stream = torch.cuda.Stream()
            own = lj.Ctx(0)
            out = torch.empty(c, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            for i in range(1500):
                lj.lj_energy_grad_batched(own, inputs[k], out, None, n_cand=c, uniform_n=n,
                                          prec=prec, stream=stream)
                if i % 50 == 0:
                    stream.synchronize()
            stream.synchronize()
            assert np.array_equal(out.cpu().numpy(), want[k])
            own.close()
        except BaseException as err:  # noqa: BLE001 -- told by the main thread
            errors.append(err)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1, 0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
