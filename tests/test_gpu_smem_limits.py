"""A kernel's dynamic shared memory limit belongs to the kernel, not to the host thread: a thread
that solves a small problem must not take back what another thread's larger problem needs."""
import threading

import pytest

from paper_1012_5379_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,large,small", [(3, 255, 47), (2, 127, 63)])
def test_a_small_problem_on_another_thread_leaves_the_limit(dim, large, small):
    from paper_1012_5379_gb300 import build, helm
    build.build()
    helm.load()

    def apply(n):
        h = helm.Handle(dim, n, 0.35, k=0.2 * (n + 1), precision="c64", maxit=1)
        r = torch.from_numpy(I.random_source(dim, n, 3)).cuda().to(torch.complex64)
        z = torch.empty_like(r)
        h.precond_apply(r, z)
        torch.cuda.synchronize()
        h.close()
        return z

    want = apply(large)
    t = threading.Thread(target=apply, args=(small,))
    t.start()
    t.join()
    assert torch.equal(apply(large), want)
