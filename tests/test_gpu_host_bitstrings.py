"""Upload of bitstrings given as Python integers: only page-locked memory is copied without a wait,
and none during stream capture."""
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# up to 256 words go as kernel parameters
@pytest.mark.parametrize("rows,cols,batch", [(3, 3, 5), (8, 9, 5), (8, 9, 128), (8, 9, 129), (3, 3, 256), (3, 3, 257)])
def test_copies_without_a_wait_are_page_locked(monkeypatch, rows, cols, batch):
    p = q.Plan(cg.grid_circuit(rows, cols, 4, 1))
    xs = cg.random_bitstrings(rows * cols, batch, 2)
    want = p.amplitude(torch.tensor(q.bitstring_words(xs, p.words), dtype=torch.int64, device="cuda"))
    unwaited, plain = [], torch.Tensor.to

    def to(self, *args, **kw):
        if kw.get("non_blocking") and not self.is_cuda:
            unwaited.append(self.is_pinned())
        return plain(self, *args, **kw)

    monkeypatch.setattr(torch.Tensor, "to", to)
    got = [p.amplitude(xs) for _ in range(50)]   # many in flight, each with its own words
    other = [p.amplitude([x ^ 1 for x in xs]) for _ in range(50)]
    monkeypatch.undo()
    assert all(unwaited) and bool(unwaited) == (batch * p.words > 256)
    assert all(torch.equal(g, want) for g in got)
    assert all(torch.equal(o, other[0]) for o in other) and not torch.equal(other[0], want)


def test_uploaded_words():
    for n in (1, 255, 256, 257, 1000):
        words = torch.randint(-(1 << 62), 1 << 62, (n,), dtype=torch.int64)
        out = torch.full((n + 1,), 7, dtype=torch.int64, device="cuda")
        host = words.clone()
        assert q.lib().qvx_words_upload(host.data_ptr(), n, out.data_ptr(), torch.cuda.current_stream().cuda_stream) == q.QVX_OK
        host.zero_()   # free to the caller at once
        assert torch.equal(out[:n].cpu(), words) and int(out[n]) == 7


@pytest.mark.parametrize("count", [2, 300])
def test_no_upload_during_capture(count):
    p = q.Plan(cg.grid_circuit(3, 3, 4, 1))
    bits = torch.tensor([1, 2], dtype=torch.int64, device="cuda")
    want = p.amplitude(bits)
    ws = p.workspace(count)
    for validate in (True, False):
        g = torch.cuda.CUDAGraph()
        with pytest.raises(q.QvxError):
            with torch.cuda.graph(g):
                p.amplitude([1, 2] * (count // 2), workspace=ws, validate=validate)
    replay, out = p.graphed(bits)
    replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
