"""Lanes per ray of a small ring's trace by what shares the GPU: the tables are the same to the bit
with one, two, four and eight lanes in every form of the medium, and a batch of many small rings
does not pay for lanes that only a ring alone can use."""
import numpy as np
import pytest
import torch

from paper_2211_00316_gb300 import phantoms as P
from paper_2211_00316_gb300 import rbx

pytestmark = pytest.mark.gpu


def make(n, nx, ny, seed, lossy=False, raw=False):
    g = P.Geometry(nx=nx, ny=ny, dx=0.9e-3, n_xducers=n, ring_radius=(min(nx, ny) - 1) * 0.45e-3 - 3e-3)
    true = P.breast_phantom(g, seed)
    job = rbx.Job()
    job.set_geometry(g, precision=rbx.RBX_BF16)
    if lossy:
        job.set_absorption(torch.tensor(P.absorption_map(true), dtype=torch.float32, device="cuda"))
    job.set_integration(raw)
    return job, torch.tensor(P.blur(true, g.dx), dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("lossy,raw", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("n,nx,ny", [(64, 96, 96), (95, 83, 110), (128, 150, 133), (190, 120, 120)])
def test_tables_same_bits(n, nx, ny, lossy, raw):
    """An update that the caller waits for has the GPU to itself; a trace that is only queued counts
    every job: beside one of 1000 transducers it takes one lane per ray."""
    job, model = make(n, nx, ny, n, lossy, raw)
    job.set_model(model)
    job.update_frequency(4e5, 1e5, torch.zeros((n, n), dtype=torch.complex64, device="cuda"))
    alone = {k: v.cpu().numpy() for k, v in job.get_tables().items()}
    large = rbx.Job()
    large.set_geometry(P.Geometry(nx=40, ny=40, dx=1e-3, n_xducers=1000, ring_radius=16e-3))
    job.set_model(model)
    job.trace_rays(4e5)
    shared = {k: v.cpu().numpy() for k, v in job.get_tables().items()}
    large.close()
    job.close()
    for k in alone:
        np.testing.assert_array_equal(alone[k], shared[k], err_msg=k)


@pytest.mark.parametrize("n,nx,jobs,limit", [(64, 96, 24, 1.9), (128, 160, 24, 1.7), (192, 200, 8, 1.22)])
def test_batch_of_small_rings(n, nx, jobs, limit):
    """The grouped form traces every ring with one lane per ray; measured, the per-job form takes 1.28,
    1.12 and 1.0 times its time with one lane, 2.8, 2.5 and 1.48 times with those of a ring alone. The
    limits lie between."""
    made = [make(n, nx, nx, s) for s in range(jobs)]
    data = [torch.view_as_complex(torch.full((2, n, n, 2), 1e-3, device="cuda")) for _ in made]
    ms = {}
    for grouped in (False, True, False, True, False, True):
        for job, model in made:
            job.set_model(model)
        _, t = rbx.batch_run([j for j, _ in made], [np.array([4e5, 5e5])] * jobs, data, grouped=grouped)
        ms[grouped] = min(t, ms.get(grouped, t))
    for job, _ in made:
        job.close()
    assert ms[False] <= limit * ms[True], ms


@pytest.mark.parametrize("n,nx", [(215, 80), (215, 96)])
def test_rings_of_thin_tubes(n, nx):
    """Where a ray's tube holds hardly a node, lanes share out nothing: alone, the trace may take no longer than
    with the one lane that it takes beside a large job (measured with two lanes: 1.40 and 1.34 times)."""
    job, model = make(n, nx, nx, n)
    data = torch.zeros((n, n), dtype=torch.complex64, device="cuda")
    job.set_slot_timing()
    large = rbx.Job()
    large.set_geometry(P.Geometry(nx=40, ny=40, dx=1e-3, n_xducers=1000, ring_radius=16e-3))
    alone, one = [], []
    for _ in range(9):
        job.set_model(model)
        alone.append(job.update_frequency(4e5, 1e5, data)["ms_kernel"]["trace"])
        job.set_model(model)
        job.update_frequency_async(4e5, 1e5, data, 0)
        one.append(job.get_stats(0)["ms_kernel"]["trace"])
    large.close()
    job.close()
    assert np.median(alone) <= 1.15 * np.median(one), (alone, one)
