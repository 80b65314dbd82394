"""The allocation-free fields where the load and the split can go wrong: rows that are no multiple of
4, 16 or 128, unaligned operands, every split of the columns, an output that overlaps an operand.
h = J s is a sum of integers: equal."""
import numpy as np
import pytest

import sg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1, 4])
@pytest.mark.parametrize("n,R", [(2, 16), (15, 16), (127, 48), (129, 16), (257, 32), (514, 80), (1001, 112),
                                 (1031, 128), (1920, 16), (2047, 128)])
def test_fields(n, R, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_11195_gb300 as sg
    rng = np.random.default_rng(n)
    J = sg_inputs.sk_couplings(n, n).astype(np.int8)
    J[rng.random((n, n)) < 0.1] = 0  # any int8 counts by its sign
    J[rng.random((n, n)) < 0.1] *= 5
    s = rng.integers(0, 2, (R, n), dtype=np.int8) * 2 - 1
    Jd = torch.zeros(n * n + 8, dtype=torch.int8, device="cuda")
    sd = torch.zeros(R * n + 8, dtype=torch.int8, device="cuda")
    Jd[offset:offset + n * n] = torch.from_numpy(J.ravel())
    sd[offset:offset + R * n] = torch.from_numpy(s.ravel())
    h = torch.full((R, n), -7, dtype=torch.int32, device="cuda")
    sg.sg_sk_fields_noalloc(Jd.data_ptr() + offset, sd.data_ptr() + offset, n, R, h.data_ptr(), 0)
    exact = s.astype(np.int64) @ np.sign(J).astype(np.int64).T
    assert np.array_equal(h.cpu().numpy(), exact)


def test_output_over_the_spins():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_11195_gb300 as sg
    n, R = 700, 32
    J = sg_inputs.sk_couplings(n, 3).astype(np.int8)
    s = np.random.default_rng(1).integers(0, 2, (R, n), dtype=np.int8) * 2 - 1
    Jd = torch.from_numpy(J).cuda()
    buf = torch.zeros(R * n, dtype=torch.int32, device="cuda")
    buf.view(torch.int8)[:R * n] = torch.from_numpy(s.ravel()).cuda()
    sg.sg_sk_fields_noalloc(Jd.data_ptr(), buf.data_ptr(), n, R, buf.data_ptr(), 0)
    assert np.array_equal(buf.cpu().numpy().reshape(R, n), s.astype(np.int64) @ J.astype(np.int64).T)
