"""oz2_dgemm splits the residue GEMM by its own estimate, not by oz2_plan's: the
same bits as oz2_dgemm_ex, which keeps to the plan, where the two take different
parts -- a split where the plan makes none, none where it makes one, and other
parts than planned.  Whether oz2_dgemm splits shows in its launches: a split's
fold is one more, a split "+1" pass's row maxima too (made from 36 saved k-blocks
on), and the fallback lists, a kernel of oz2_dgemm_ex, are one less."""
import pytest

from helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def oz():
    ensure_built()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_06510_gb300 as oz
    oz.lib()
    return oz


@pytest.mark.parametrize("m,n,k,r,planned,split", [
    (515, 81, 3815, 13, 2, False),      # 2 planned, none taken
    (1282, 86, 4663, 13, 1, True),      # none planned, 2 taken
    (1040, 651, 47202, 8, 1, True),     # none planned, 5 taken
    (900, 800, 40000, 10, 2, True),     # 2 planned, 4 taken
    (1306, 170, 35472, 8, 6, True),     # 6 planned, 3 taken
    (622, 341, 36468, 12, 2, False),    # 2 planned, none taken
    (197, 130, 6151, 6, 5, True),       # 5 planned, 6 taken
])
def test_same_bits_as_the_planned_call(oz, m, n, k, r, planned, split):
    import torch
    plan = oz.oz2_plan(m, n, k, r)
    assert plan["kparts"] == planned
    blocks, parts = (k + 127) // 128, plan["mag_kparts"]
    own_sums = parts > 1 and blocks - (blocks + parts - 1) // parts >= 36
    g = torch.Generator(device="cuda")
    g.manual_seed(600 + m)
    A = torch.randn((k, m), dtype=torch.float64, device="cuda", generator=g).exp_().t() - 1.0
    B = torch.randn((n, k), dtype=torch.float64, device="cuda", generator=g).exp_().t() - 1.0
    A, B = oz.colmajor(A), oz.colmajor(B)

    def launches(call):
        call()
        oz.oz2_get_stats()
        got = call()
        return got, oz.oz2_get_stats()["kernel_launches"]

    (want, _), ex = launches(lambda: oz.oz2_dgemm_ex(A, B, num_moduli=r))
    got, own = launches(lambda: oz.oz2_dgemm(A, B, num_moduli=r))
    assert torch.equal(got.t().contiguous().view(torch.int64), want.t().contiguous().view(torch.int64))
    assert own - (ex - 1) == int(split) - int(planned > 1) + int(own_sums) - int(parts > 1)
    assert oz.oz2_check_device_status() == 0
