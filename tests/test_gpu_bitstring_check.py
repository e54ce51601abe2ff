"""Device bitstring checks: what is refused, that a refused call leaves the caller's memory and
angles as they were, other streams, threads, and stream capture."""
import threading

import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def words(xs, p):
    return torch.tensor(q.bitstring_words(xs, p.words), dtype=torch.int64, device="cuda")


@pytest.mark.parametrize("rows,cols,bad_bit", [(3, 3, 9), (3, 3, 63), (8, 9, 72), (8, 9, 127)])
@pytest.mark.parametrize("count", [1, 300, 20000])
def test_refused(rows, cols, bad_bit, count):
    p = q.Plan(cg.grid_circuit(rows, cols, 4, 1))
    ok = p.amplitude(words([1, 2, 3], p))
    xs = [0] * count
    xs[count // 2] = 1 << bad_bit
    bits = words(xs, p)
    for call in (p.amplitude, p.slice_terms):
        with pytest.raises(q.QvxError):
            call(bits)
    out = torch.full((2 * count,), 7.0, dtype=torch.float64, device="cuda")
    with pytest.raises(q.QvxError):
        p.amplitude(bits, out=out)
    assert bool((out == 7.0).all())
    assert torch.equal(p.amplitude([1, 2, 3]), ok) and torch.equal(p.amplitude(words([1, 2, 3], p)), ok)


def test_refused_gradient_keeps_the_angles():
    c = cg.rotation_circuit(2, 3, 4, 44)
    p = q.Plan(c, gradient=True)
    ws = p.workspace(1)
    th = torch.tensor(c.thetas(), dtype=torch.float64, device="cuda")
    p.amplitude_grad([5], th, workspace=ws)
    want = p.amplitude([5], workspace=ws)
    with pytest.raises(q.QvxError):
        p.amplitude_grad(words([1 << 6], p), th + 1.0, workspace=ws)
    assert torch.equal(p.amplitude([5], workspace=ws), want)


def test_other_stream_and_threads():
    p = q.Plan(cg.grid_circuit(4, 4, 10, 1001), n_slices=2)
    xs = cg.random_bitstrings(16, 8, 3)
    want = p.amplitude(xs)
    s = torch.cuda.Stream()
    bits = torch.zeros(8, dtype=torch.int64, device="cuda")
    for _ in range(20):   # bitstrings written on the current stream, work on another one
        bits.zero_()
        bits.copy_(words(xs, p))
        got = p.amplitude(bits, stream=s)
        s.synchronize()
        assert torch.equal(got, want)
    failures = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ws = p.workspace(8)
                for k in range(50):
                    b = words(xs, p)
                    if (k + i) % 3 == 0:
                        b[k % 8] = 1 << 40
                        try:
                            p.amplitude(b, workspace=ws)
                            failures.append("not refused")
                        except q.QvxError:
                            pass
                    elif not torch.equal(p.amplitude(b, workspace=ws), want):
                        failures.append("wrong")
        except Exception as e:   # reported in the main thread
            failures.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures[:3]


def test_no_check_during_capture():
    p = q.Plan(cg.grid_circuit(3, 3, 4, 1))
    bits = words([1, 2], p)
    p.amplitude(bits)
    g = torch.cuda.CUDAGraph()
    with pytest.raises(q.QvxError):
        with torch.cuda.graph(g):
            p.amplitude(bits)
    replay, out = p.graphed(bits)
    replay()
    torch.cuda.synchronize()
    assert torch.equal(out, p.amplitude([1, 2]))
