"""Host threads that each use a state of their own: what one thread's launches set on a
kernel must not reach another thread's launches."""

import threading

import numpy as np
import pytest

from test_gpu_parity import setup_case

pytestmark = pytest.mark.gpu


def in_threads(jobs):
    """Run every job in a thread of its own, all started together; their exceptions."""
    errors, gate = [], threading.Barrier(len(jobs))

    def run(job):
        try:
            gate.wait()
            job()
        except Exception as e:
            errors.append(e)
    threads = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


# grids whose double-precision stress tiles differ in shape and so in shared memory:
# 32 x 4, 18 x 7 and 64 x 2 columns
@pytest.mark.parametrize("model,extra", [('oldroyd_b', {}), ('saramito', {'Bi': 0.4})])
def test_double_precision_stress_from_several_threads(evp, model, extra):
    import torch
    sims = [setup_case(evp, s, model, extra, evp.EVP_FP64)[0] for s in
            ((32, 32, 8, False), (72, 54, 8, False), (128, 6, 8, True))]
    outs = [torch.empty((6,) + s.shape, dtype=torch.float64, device='cuda') for s in sims]
    want = []
    for s, o in zip(sims, outs):
        evp.evp_stress_rhs(s.handle, o)
        s.sync()
        want.append(o.cpu().numpy())

    lib = evp.load()

    def job(s, p):
        def repeat():
            for _ in range(3000):          # the bare call: little else between a thread's launches
                assert lib.evp_stress_rhs(s.handle, p) == 0, evp.evp_last_error()
            s.sync()
        return repeat
    assert not in_threads([job(s, o.data_ptr()) for s, o in zip(sims, outs)])
    for w, o in zip(want, outs):
        assert np.array_equal(w, o.cpu().numpy())


# lines of 216, 384 and 512 points, whose column passes differ in shared memory beyond the
# default limit
@pytest.mark.parametrize("prec", [0, 1])
def test_poisson_solves_from_several_threads(evp, prec):
    import torch
    sims = [setup_case(evp, (8, 8, nz, False), 'newtonian', {}, prec)[0] for nz in (216, 384, 512)]
    rhs, psi, want = [], [], []
    for s in sims:
        r = torch.randn(s.shape, dtype=s.dtype, device='cuda', generator=torch.Generator('cuda').manual_seed(1))
        rhs.append(r - r.mean())
        psi.append(torch.empty_like(r))
        evp.evp_poisson_solve(s.handle, rhs[-1], psi[-1])
        s.sync()
        want.append(psi[-1].cpu().numpy())

    def job(s, r, p):
        def repeat():
            for _ in range(600):
                evp.evp_poisson_solve(s.handle, r, p)
            s.sync()
        return repeat
    assert not in_threads([job(*a) for a in zip(sims, rhs, psi)])
    for w, p in zip(want, psi):
        assert np.array_equal(w, p.cpu().numpy())
