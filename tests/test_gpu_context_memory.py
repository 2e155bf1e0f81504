"""Contexts, batches and networks give back all the device memory they took."""
import pytest

pytestmark = pytest.mark.gpu


def test_memory_is_given_back():
    import torch

    import paper_1610_05258_gb300 as pmt
    from paper_1610_05258_gb300 import workloads as W

    inst = W.uniform_instance(64, 4, F=2, seed=1)
    px, py, v = (torch.from_numpy(a).cuda() for a in (inst.px, inst.py, inst.vals))
    hx, hy, hv = (t.cpu().pin_memory() for t in (px, py, v))
    out, mesh = torch.empty(2, 4096, device="cuda"), torch.empty(2, 4096).pin_memory()

    def use():
        for dim, kind in ((2, "q1"), (2, "p1"), (1, "q1")):
            c = pmt.Context(dim, 64, 1.0, inst.np, 2, mesh=kind)
            if dim == 2:
                c.assign_mass(px, py, v, out=out)
                c.assign_mass_host(hx, hy, hv, out=mesh)
        c = pmt.Context(2, 128, 1.0, inst.np, 2)  # with the network's arrays
        net = pmt.Net(128, 2)
        b = pmt.Batch([64, 32], [1.0, 1.0], [inst.np, 100], 2)
        del c, net, b
        torch.cuda.synchronize()

    for _ in range(3):
        use()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(20):
        use()
    # a leak of one allocation in every round would be 20 times its 2 MB granule
    assert torch.cuda.mem_get_info()[0] >= free - 20 * (1 << 20)
