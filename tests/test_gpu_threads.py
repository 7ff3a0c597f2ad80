"""One handle per host thread: calls of different sizes made at the same time."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,G,ranks", [
    (4864, 512, (64, 32)),   # 64 x 128 tiles: 49 and 25 KiB of shared memory, 48 KiB need no opt-in
    (512, 136, (128, 8)),    # 64 x 64 tiles: 66 and 4 KiB
])
def test_adapter_projections_of_two_threads(N, G, ranks):
    """The kernels' shared-memory limit belongs to the device: the call of the smaller rank must
    not lower it between another thread's setting it and that thread's launch."""
    import paper_2609_04526_gb300 as pkg
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N)
    base = torch.randint(0x30, 0x60, (N, G), generator=gen, device="cuda", dtype=torch.uint8)
    work = []
    for r in ranks:
        B = (torch.randn(N, r, generator=gen, device="cuda") * 0.1).bfloat16()
        A = (torch.randn(r, G, generator=gen, device="cuda") * 0.1).bfloat16()
        out = torch.empty_like(base)
        h = pkg.Handle()
        h.sq_project_lowrank(pkg.NVFP4, base, B, A, 0.01, 1.0, bytes_out=out)
        h.sq_sync()
        work.append((h, B, A, out, out.clone()))
    failed = []

    def calls(h, B, A, out):
        stream = torch.cuda.Stream()
        try:
            for _ in range(4000):
                h.sq_project_lowrank(pkg.NVFP4, base, B, A, 0.01, 1.0, bytes_out=out, stream=stream)
            h.sq_sync(stream)
        except pkg.SQError as e:
            failed.append(str(e))

    threads = [threading.Thread(target=calls, args=w[:4]) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for _, _, _, out, alone in work:
        assert torch.equal(out, alone)
