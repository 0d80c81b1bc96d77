"""What a bounded wait that gives up does to the calls around it, in every precision. The wait runs
out on the job's stream (a barrier that nothing signals, about a second) and is recorded where the
contractions record theirs: stand-alone calls then give results that are not a number, an update
fails and leaves the model, each failure is reported once, and the job goes on as before."""
import numpy as np
import pytest
import torch

from paper_2211_00316_gb300 import phantoms as P
from paper_2211_00316_gb300 import rbx

pytestmark = pytest.mark.gpu

F, DF = 3e5, 1e5
ETIMEOUT = 6


def reported(call):
    with pytest.raises(rbx.RbxError) as e:
        call()
    return e.value.status == ETIMEOUT


@pytest.mark.parametrize("precision", [rbx.RBX_FP32, rbx.RBX_BF16, rbx.RBX_BF16X3])
@pytest.mark.parametrize("n,lossy", [(48, False), (200, True)])
def test_reported_once(precision, n, lossy):
    w = P.custom(n, 64, 1e-3, 28e-3, kind="discs", freqs=(F,))
    rng = np.random.default_rng(n)
    R = torch.tensor(1e-3 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))), device="cuda").to(torch.complex64)
    dm = torch.tensor(1e-9 * rng.standard_normal((64, 64)), dtype=torch.float32, device="cuda")
    model = torch.tensor(w.c_init, dtype=torch.float32, device="cuda")
    job = rbx.Job()
    job.set_geometry(w.geom, precision=precision)
    if lossy:
        job.set_absorption(torch.tensor(P.absorption_map(w.c_true), dtype=torch.float32, device="cuda"))
    job.set_model(model)
    job.trace_rays(F)
    calls = [lambda: job.forward(F, dm), lambda: job.adjoint(F, R, False), lambda: job.adjoint(F, R, True),
             lambda: job.predict(F)[~torch.eye(n, dtype=torch.bool, device="cuda")]]
    good = [c() for c in calls]
    job.sync()
    job.selftest_timeout()
    for c in calls:
        assert bool(torch.isnan(torch.view_as_real(c())).any(-1).all())
    assert reported(job.sync)
    job.sync()
    for c, want in zip(calls, good):
        assert bool((c() == want).all())

    job.selftest_timeout()
    assert reported(lambda: job.update_from_tables(F, DF, R))
    assert bool((job.get_model() == model).all())
    job.sync()
    job.update_from_tables(F, DF, R)
    updated = job.get_model()
    assert not bool((updated == model).all())

    job.set_model(model)
    job.selftest_timeout()
    assert reported(lambda: job.update_set([F, F + DF], DF, torch.stack([R, R])))
    assert bool((job.get_model() == model).all())
    job.update_frequency_async(F, DF, R, 3)
    job.get_stats(3)
    job.close()


def test_reported_from_a_graph():
    """A forward captured into the caller's graph runs again without a call of the library."""
    n = 48
    w = P.custom(n, 64, 1e-3, 28e-3, kind="discs", freqs=(F,))
    dm = torch.full((64, 64), 1e-9, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        job = rbx.Job(stream)
        job.set_geometry(w.geom, precision=rbx.RBX_FP32)
        job.set_model(torch.tensor(w.c_init, dtype=torch.float32, device="cuda"))
        job.trace_rays(F)
        want = job.forward(F, dm).clone()
        job.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            out = job.forward(F, dm)
        job.sync()
        job.selftest_timeout()
        graph.replay()
        assert reported(job.sync)
        assert bool(torch.isnan(torch.view_as_real(out)).any(-1).all())
        graph.replay()
        job.sync()
        assert bool((out == want).all())
        del graph
        job.close()
