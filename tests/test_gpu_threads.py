"""Meshes of different sizes and degrees used at the same time from several host threads."""
import threading

import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(workers):
    errors = []

    def guarded(f):
        try:
            f()
        except Exception as ex:      # a refused launch
            errors.append(str(ex))
    threads = [threading.Thread(target=guarded, args=(f,)) for f in workers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("what", ["jvp", "apply"])
def test_threads_with_small_and_large_meshes(what):
    """Two threads, each with its own mesh and stream, launch the same kernels with different amounts of dynamic
    shared memory (degree 1: 192 and 12,288 elements, one warp or four per CTA; the block-Jacobi apply:
    degrees 1 and 3). Every launch is accepted, and the results are those of the calls made alone."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    shapes = ((2, 1), (16, 1)) if what == "jvp" else ((2, 1), (2, 3))
    sets = []
    for n, p in shapes:
        d = W.shell_desc(n=n, nr=8, p=p)
        d.h_first = 0.0
        m = Mesh(d)
        u = torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()
        v = torch.from_numpy(W.normal(5, u.numel()).reshape(u.shape)).cuda()
        if what == "apply":
            m.precond_setup("bj", u, 0.2, 1e-4)
        call = (lambda m=m, u=u, v=v, o=None: m.jvp(u, v, 0.3, out=o)) if what == "jvp" else \
            (lambda m=m, v=v, o=None: m.precond_apply("bj", v, out=o))
        sets.append((m, u, call, call()))
    torch.cuda.synchronize()

    def worker(m, u, call, ref):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            out = torch.empty_like(u)
            for _ in range(4000):
                call(o=out)
            s.synchronize()
        assert torch.equal(out, ref)
    _run([lambda a=a: worker(*a) for a in sets])
    for m, *_ in sets:
        m.close()
