"""Solvers and networks of different sizes on two host threads: every call succeeds and
gives the bits of the same call made alone.  A kernel's shared-memory limit belongs to the
process, so a launch that first sets it to its own size can lower it between another
thread's set and launch."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


def _together(jobs):
    """Runs the jobs on a thread each; returns their errors."""
    errors, start = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            start.wait()
            job()
        except Exception as e:
            errors.append(repr(e))

    ts = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return errors


def _solver_job(fh, dims, prec, path, reps, stream):
    M = np.diag(dims) if len(dims) == 3 else [[dims[0], 0], [0, dims[1]]]
    d = len(dims)
    s = fh.Solver(fh.Pattern(M), fh.generator("dlvp", alpha=[0.25] * d), 1, stream)
    ids = (np.random.default_rng(3).random(s.m) < 0.2).astype(np.uint8)
    s.set_stiffness_phases(ids, np.stack([fh.isotropic_stiffness(*fh.lame(E, nu), d) for E, nu in ((1.0, 0.3), (9.0, 0.2))]))
    s.set_reference(None)
    eps0 = np.eye(s.nv)[:1]
    opts = dict(tol=0.0, max_iter=3, precision=prec, path=path)   # below a replay: single launches
    s.solve(eps0, **opts)
    ref = s.get_strain(0)

    def job():
        for _ in range(reps):
            s.solve(eps0, **opts)
        assert np.array_equal(s.get_strain(0), ref)

    return s, job


# general two-step passes, block passes and cluster solves, a large and a small grid each
@pytest.mark.parametrize("large,small,prec,path", [([1, 480, 480], [2, 20, 20], 1, 1), ([1, 240, 240], [2, 20, 20], 0, 1),
                                                   ([2, 34, 374], [2, 17, 34], 1, 1), ([160, 160], [9, 18], 1, 2)],
                         ids=["general_fp32", "general_fp64", "block_fp32", "cluster_fp32"])
def test_two_solvers_on_two_threads(fh, large, small, prec, path):
    import torch
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    a, ja = _solver_job(fh, large, prec, path, 150, streams[0].cuda_stream)
    b, jb = _solver_job(fh, small, prec, path, 600, streams[1].cuda_stream)
    assert _together([ja, jb]) == []
    a.close()
    b.close()


def test_two_networks_on_two_threads(fh):
    import torch
    nets, jobs, keep = [], [], []
    for n, width, modes, reps in ((48, 48, 12, 60), (8, 4, 2, 400)):
        st = torch.cuda.Stream()
        net = fh.FNO(n, 1, 6, width, modes, 2, max_batch=1, stream=st.cuda_stream)
        g = torch.Generator(device="cuda").manual_seed(n)
        net.set_params((0.2 * torch.randn(net.nparam, generator=g, device="cuda")).cpu().numpy())
        x = torch.randn(1, 1, n ** 3, generator=g, device="cuda")
        y = torch.empty(1, 6, n ** 3, device="cuda")
        torch.cuda.synchronize()
        net.forward(x, y)
        ref = y.clone()
        torch.cuda.synchronize()

        def job(net=net, x=x, y=y, reps=reps):
            for _ in range(reps):
                net.forward(x, y)

        nets.append(net)
        jobs.append(job)
        keep.append((y, ref))
    assert _together(jobs) == []
    for y, ref in keep:
        assert torch.equal(y, ref)
    for net in nets:
        net.close()
