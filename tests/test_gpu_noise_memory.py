"""The buffer that keeps a noisy 2D / 3D step's normals is taken only where memory is
plentiful: two problems whose fields and scratch fields just fit still run, and draw
the same noise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_problems_that_just_fit_run_without_the_noise_buffer():
    import torch
    from paper_1204_4255_gb300 import xsde
    shape, npaths = (512, 512), 128
    field = npaths * shape[0] * shape[1] * 8

    def problem():
        P = xsde.Problem(shape, (-6.0, -6.0), (6.0, 6.0), "c64")
        P.set_operators(g=1.0, pot_kind=xsde.XSDE_POT_HARMONIC, omega=(1.0, 1.0), seed=4, amplitude=0.1,
                        noise_kind=xsde.XSDE_NOISE_WIENER_COMPLEX)
        return P

    def psi():
        x = torch.linspace(-6.0, 6.0, 513, device="cuda")[:-1]
        return torch.exp(-0.5 * (x[:, None] ** 2 + x ** 2)).to(torch.complex64).expand(npaths, *shape).contiguous()

    # with memory to spare (and the kernels loaded)
    P = problem()
    want = psi()
    P.integrate(want, 1e-4, 3)
    P.synchronize()
    P.close()
    want = want.cpu().numpy()
    fields = [psi(), psi()]
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - int(2.6 * field), dtype=torch.uint8, device="cuda")
    problems = [problem(), problem()]
    try:
        for P, x in zip(problems, fields):
            P.integrate(x, 1e-4, 3)
            P.synchronize()
    finally:
        for P in problems:
            P.close()
        del hold
        torch.cuda.empty_cache()
    for x in fields:
        got = x.cpu().numpy()
        assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-6
