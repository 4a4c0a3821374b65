"""Batched solves of different sizes from several host threads: each thread's
calls are accepted and give what they give alone."""
import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch


# sizes that take the same kernel with different amounts of shared memory
@pytest.mark.parametrize("method", ["ONCHIP", "GLOBAL", "GLOBAL_FMA"])
def test_threads_with_different_sizes(torch, method):
    from paper_1110_4903_gb300 import chem
    which = getattr(chem, "LU_" + method)
    systems, sizes = 8, (60, 100, 61, 150)
    gen = torch.Generator().manual_seed(5)

    def solve(case):
        A0, b0, A, b = case
        A.copy_(A0)
        b.copy_(b0)
        chem.batched_solve(which, A, b)

    cases = []
    for n in sizes:
        A = torch.randn((systems, n, n), generator=gen, dtype=torch.float64) + n ** 0.5 * torch.eye(n, dtype=torch.float64)
        b = torch.randn((systems, n), generator=gen, dtype=torch.float64)
        if method != "ONCHIP":
            A, b = A.permute(1, 2, 0).contiguous(), b.T.contiguous()
        A, b = A.cuda(), b.cuda()
        cases.append((A, b, torch.empty_like(A), torch.empty_like(b)))
    alone = []
    for c in cases:
        solve(c)
        alone.append((c[2].clone(), c[3].clone()))
    torch.cuda.synchronize()
    start, errors = threading.Barrier(len(sizes)), []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                start.wait()
                for _ in range(1500):
                    solve(cases[i])
                stream.synchronize()
        except Exception as exc:
            errors.append((sizes[i], str(exc)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for c, (A, b) in zip(cases, alone):
        assert torch.equal(c[2], A) and torch.equal(c[3], b)
