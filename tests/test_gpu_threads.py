"""Host threads that recover on lattices of different length at once, on streams
of their own: the transforms share kernels whose shared memory they need in
different sizes, and every call returns what it returns alone."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [(2**22, 2**20), (2**23, 3 * 2**21), (10**6, 4 * 10**6)])
def test_recoveries_of_two_lengths(lengths):
    from paper_2302_00752_gb300 import binding as B

    def inputs(M):
        rng = np.random.default_rng(M)
        k = rng.choice(np.arange(1, M // 2 - 1), 8, replace=False)[:, None]
        c = rng.standard_normal(8) + 1j * rng.standard_normal(8)
        cand = torch.as_tensor(np.vstack([k, -k]).astype(np.int32)).cuda()
        return M, torch.as_tensor(k.astype(np.int32)).cuda(), torch.as_tensor(c).cuda(), cand

    data = [inputs(M) for M in lengths]
    ref = [B.sft_recover([1], *d)[1].clone() for d in data]
    torch.cuda.synchronize()
    fails = []

    def work(d, want):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for _ in range(100):
                    v = B.sft_recover([1], *d)[1]
                    st.synchronize()
                    assert torch.equal(v, want)
        except Exception as e:
            fails.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in zip(data, ref)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not fails
