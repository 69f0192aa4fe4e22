"""Host threads that call the library at once, each with its own stream,
workspace and sizes: a kernel's attributes are shared by all of them."""
import os
import re
import threading

import pytest

torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1301_1071_gb300", "csrc")


def test_one_shared_memory_attribute_per_function():
    """Only allow_smem sets a function's largest dynamic shared memory, and to a
    value that does not follow the call's sizes: a thread that set its own (smaller)
    size could lower it between another's setting and launch, which then fails."""
    uses = []
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        uses += [f] * len(re.findall(r"cudaFuncSetAttribute", src))
    assert uses == ["launch.h"]
    src = open(os.path.join(CSRC, "launch.h")).read()
    body = src[src.index("inline cudaError_t allow_smem"):]
    body = body[:body.index("\n}")]
    assert re.search(r"MaxDynamicSharedMemorySize, static_cast<int>\(most\)\)", body)
    assert "bytes" not in body[body.index("cudaFuncSetAttribute"):]


@pytest.mark.gpu
def test_threads_with_different_sizes():
    import paper_1301_1071_gb300 as T
    sizes = [(20_000, 8), (3_000, 64), (5_000, 25), (2_000, 50)]
    inputs = {}
    for k, (m, n) in enumerate(sizes):
        g = torch.Generator(device="cuda").manual_seed(40 + k)
        for dt in (torch.float64, torch.float32):
            A = torch.randn(m, n, dtype=dt, device="cuda", generator=g)
            inputs[k, dt] = (A, T.direct(A), T.cholqr(A), T.r(A))
    torch.cuda.synchronize()
    errors = []

    def work(k, dt):
        try:
            s = torch.cuda.Stream()
            A, (Q, R), (Qc, Rc), Rr = inputs[k, dt]
            with torch.cuda.stream(s):
                for _ in range(150):
                    q, r = T.direct(A, check=False)
                    qc, rc = T.cholqr(A, check=False)
                    rr = T.r(A, check=False)
                s.synchronize()
                assert torch.equal(q, Q) and torch.equal(r, R)
                assert torch.equal(qc, Qc) and torch.equal(rc, Rc) and torch.equal(rr, Rr)
        except Exception as e:  # noqa: BLE001 -- reported below, by the main thread
            errors.append((sizes[k], dt, repr(e)[:200]))

    threads = [threading.Thread(target=work, args=kd) for kd in inputs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
