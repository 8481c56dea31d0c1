"""Host-resident depth-0 products of less than a wave of tiles: two panels only where
what they hide is more than the second panel's wave.  A C in A's memory is always one
panel, so its time stands for one."""
import pytest

pytestmark = pytest.mark.gpu


# long K: 236 us in one panel, 325 in two
@pytest.mark.parametrize("m,n,k", [(656, 117, 4288), (64, 448, 3568)])
def test_a_second_wave_is_not_taken_for_little(m, n, k):
    import torch
    from paper_1205_2927_gb300 import fmm
    A, B = torch.rand(m, k).pin_memory(), torch.rand(k, n).pin_memory()
    own, shared = torch.empty(m, n).pin_memory(), A.view(-1)[: m * n].view(m, n)
    p = fmm.Plan(m, n, k, depth=0, leaf_tile=256, host_operands=1, host_copy="sm")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ms = []
    for C in (own, shared):
        runs = []
        for _ in range(6):
            e[0].record()
            for _ in range(10):
                p(A, B, C)
            e[1].record()
            torch.cuda.synchronize()
            runs.append(e[0].elapsed_time(e[1]) / 10)
        ms.append(min(runs[1:]))
    p.close()
    assert ms[0] <= 1.2 * ms[1], ms
