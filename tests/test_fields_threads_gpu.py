"""The allocation-free SK fields from several host threads at once, each on a stream of its own with inputs of
its own: integers equal to the matrix product."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_calls_of_several_threads_overlap():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_11195_gb300 as sg
    jobs = []
    for k, (n, R) in enumerate([(2000, 128), (129, 16), (777, 48), (2048, 128), (64, 16), (1500, 64)]):
        g = torch.Generator(device="cuda").manual_seed(k)
        J = torch.randint(0, 2, (n, n), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
        s = torch.randint(0, 2, (R, n), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
        want = (s.double() @ J.double().T).to(torch.int32)
        jobs.append((J, s, want, torch.empty_like(want), torch.cuda.Stream(), []))
    torch.cuda.synchronize()

    def work(J, s, want, h, stream, errors):
        try:
            for _ in range(30):
                with torch.cuda.stream(stream):
                    h.fill_(-1)
                sg.sg_sk_fields_noalloc(J.data_ptr(), s.data_ptr(), J.shape[0], s.shape[0], h.data_ptr(),
                                        stream.cuda_stream)
                with torch.cuda.stream(stream):
                    if not torch.equal(h, want):
                        errors.append("fields differ")
        except Exception as e:  # reported by the test's own thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not [e for j in jobs for e in j[5]]
