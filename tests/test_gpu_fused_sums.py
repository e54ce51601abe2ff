"""The fused engine's sums of the item partials, by the block or a warp for each amplitude: bit for
bit the sum of one amplitude alone, and NaN for the whole call where one is outside the range."""
import numpy as np
import pytest

import circuitgen as cg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# 1, 16, 128 and 1024 partials an amplitude; batches around the warps of a block (1 to 32)
@pytest.mark.parametrize("k,inner,warps,opened", [(0, 0, 1, []), (4, 0, 4, [3]), (7, 0, 8, []), (10, 0, 1, []), (10, 0, 16, [0, 7])])
@pytest.mark.parametrize("batch", [1, 2, 7, 24, 25, 33, 200])
def test_batches_equal_single_amplitudes(k, inner, warps, opened, batch):
    n = 16
    p = q.Plan(cg.grid_circuit(4, 4, 14, 77), n_slices=k, inner_slices=inner, warps_per_item=warps, engine="fused",
               open_qubits=opened)
    xs = cg.random_bitstrings(n, batch, 5)
    got = p.amplitude(xs)
    for b in {0, batch // 2, batch - 1}:
        assert torch.equal(got[b], p.amplitude([xs[b]])[0])
    # the stepwise engine adds the same terms exactly, in any order
    other = q.Plan(cg.grid_circuit(4, 4, 14, 77), order=p.order, slices=p.slices, inner_slices=inner, engine="stepwise",
                   open_qubits=opened)
    assert float((got - other.amplitude(xs)).abs().max()) < 1e-5 * 2.0 ** (-n / 2)


@pytest.mark.parametrize("batch", [2, 40])
def test_out_of_range_amplitudes_make_the_call_nan(batch):
    # diag(2^28, 1) on qubit 0: only amplitudes with that bit 0 are outside the exact sum's range
    c = cg.Circuit(2, [cg.Gate(cg.H, 0), cg.Gate(cg.H, 1), cg.Gate(cg.CZ, 0, 1),
                       cg.Gate(cg.U1, 0, u=(2.0 ** 30, 0, 0, 0, 0, 0, 1.0, 0)), cg.Gate(cg.H, 1)])
    p = q.Plan(c, engine="fused", host_merge_rank=0)
    ws = p.workspace(batch)
    fine = p.amplitude([1] * batch, workspace=ws).cpu().numpy()
    assert np.isfinite(fine).all()
    got = p.amplitude([1] * (batch - 1) + [0], workspace=ws).cpu().numpy()
    assert np.isnan(got).all()
    with pytest.raises(q.QvxError) as e:
        p.check_status(ws)
    assert e.value.status == q.QVX_ERANGE
    assert np.array_equal(p.amplitude([1] * batch, workspace=ws).cpu().numpy(), fine)
