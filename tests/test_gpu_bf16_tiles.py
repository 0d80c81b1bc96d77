"""The BF16 operand synthesis in tiles of 32 and of 64 transducers (the count decides), at counts around
their edges and odd node counts: forward, preconditioned adjoint and the norm of an update's step against the
FP32 job on the same tables. Each operand is rounded to BF16 (2^-9 at most): two in the forward, three
in the adjoint (u, R and the weights), 3 x 2^-9 = 5.9e-3 of every product at most."""
import numpy as np
import pytest
import torch

from paper_2211_00316_gb300 import phantoms as P
from paper_2211_00316_gb300 import rbx
from test_gpu_fp32_contractions import F, rel, tables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 33, 63, 64, 65, 66, 95, 97, 100, 127, 128, 129, 161, 192, 193, 449, 513])
def test_against_fp32(n):
    g = P.Geometry(nx=41, ny=37, dx=1e-3, n_xducers=n, ring_radius=16.5e-3)
    T, a, gam, K = tables(g, n)
    rng = np.random.default_rng(n)
    R = torch.tensor(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)), device="cuda").to(torch.complex64)
    dm = torch.tensor(1e-9 * rng.standard_normal((37, 41)), dtype=torch.float32, device="cuda")
    out = {}
    for precision in (rbx.RBX_FP32, rbx.RBX_BF16):
        job = rbx.Job()
        job.set_geometry(g, precision=precision)
        job.set_tables(*[torch.tensor(t, device="cuda") for t in (T, a, gam, K)], torch.zeros((n, n - 1, 4), device="cuda"))
        out[precision] = [job.forward(F, dm).cpu().numpy(), job.adjoint(F, R, True).cpu().numpy()]
        # one pass over the tables writes both contractions' operands; the step's norm as the update reports it
        # (the model keeps the step to its own FP32 quantum only)
        out[precision].append(np.array([job.update_from_tables(F, 1e5, 1e-6 * R)["dm_norm"]]))
        job.close()
    for x, y in zip(out[rbx.RBX_BF16], out[rbx.RBX_FP32]):
        assert rel(x, y) <= 5.9e-3
