"""Several host threads running layers of different sizes through the same
kernels: a launch needs the shared memory of its own plan whatever another
thread's launch, or planning, of the same kernel asked for in between."""
import threading

import pytest
import torch

import paper_1512_06473_gb300 as q
from paper_1512_06473_gb300 import _lib

pytestmark = pytest.mark.gpu

# N, Cs, H, Ct, k, pad: each pair through one kernel with unlike plans
PAIRS = {
    "contract": [(1, 8, 5, 8, 3, 1), (4, 64, 28, 130, 3, 1)],
    "contract_1x1": [(1, 8, 4, 8, 1, 0), (8, 128, 14, 200, 1, 0)],
    "chunked": [(1, 8, 5, 8, 3, 1), (2, 32, 40, 130, 3, 1)],
}


@pytest.mark.parametrize("name", list(PAIRS))
def test_launches_of_one_kernel_from_several_threads(name):
    algo = name.split("_")[0]
    g = torch.Generator(device="cuda").manual_seed(11)
    jobs, keep = [], []
    for N, Cs, H, Ct, k, pad in PAIRS[name] * 2:
        x = torch.randn((N, Cs, H, H), generator=g, device="cuda")
        D = torch.randn((Cs // 4, 16, 4), generator=g, device="cuda")
        c = torch.randint(0, 16, (Ct, k * k, Cs // 4), generator=g, device="cuda",
                          dtype=torch.uint8)
        want = q.conv_forward(x, D, c, k, k, 1, pad, algo=algo)
        out, ws = torch.empty_like(want), torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
        st = torch.cuda.Stream()
        args = (x.data_ptr(), N, Cs, H, H, Ct, k, k, 1, pad, D.data_ptr(), 4, 16, c.data_ptr(), 0,
                None, out.data_ptr(), 0, _lib.ALGO[algo], 0, ws.data_ptr(), ws.numel(),
                st.cuda_stream)
        jobs.append((args, want, out, st))
        keep.append((x, D, c, ws))
    torch.cuda.synchronize()
    bad = []
    start = threading.Barrier(len(jobs))
    forward = q.load().qcnn_conv_forward

    def work(args):
        torch.cuda.set_device(0)
        start.wait(30)
        for _ in range(2000):
            rc = forward(*args)
            if rc:
                bad.append(rc)

    threads = [threading.Thread(target=work, args=(j[0],)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad, (len(bad), bad[0])
    for _, want, out, _ in jobs:
        assert torch.equal(out, want)
