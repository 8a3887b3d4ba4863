"""lbcg_step_launches counts the kernels that a call of the resident kernel's length launches."""
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("n", [8, 31, 33, 64])
def test_launches_of_one_resident_call(prec, n):
    # one cooperative launch; in 16-bit storage a second kernel advances the count of graph replays
    # that the call stands for, where it stands for any
    from paper_1707_00198_gb300.lbcg import Lattice
    g, p = I.config_static_droplet()
    L = Lattice(g, p, prec)
    L.set_tile(8)
    for pool in (0, n & 1):
        before = L.step_launches
        L.step(n)
        # (from the second pool a call takes one step before its replays)
        assert L.step_launches - before == 1 + (prec in ("fp16", "bf16") and (n - pool) // 32 > 0)
    L.close()
