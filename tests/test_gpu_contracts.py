"""What the entry points promise beside their results: pointers they take,
stages they mark, tile shapes they keep to, and paths that only wide or
unevenly split tables reach.  Every result equals the CPU oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import ensure_built
from paper_1202_1350_gb300 import vc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P = (1 << 61) - 1


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, np.uint64)).view(np.int64).copy()).cuda()


def elements(seed, n):
    """n field elements over the whole range, both ends among them."""
    x = oracle.splitmix64(seed, n) >> np.uint64(3)
    x[x == P] = 0
    x[::7] = P - 1
    x[3::11] = 0
    return x


# a proof buffer at any byte of device memory, as a copy takes it
@pytest.mark.parametrize("offset", [0, 1, 4, 8, 12])
def test_f2sp_proof_at_any_byte(offset):
    v, h = 19, 13
    a = elements(offset, v * h)
    want = oracle.f2sp_prove(a, v, h)
    buf = torch.full((16 * h + 32,), 0x5A, dtype=torch.uint8, device="cuda")
    s = vc.vc_f2sp_create(v, h)
    try:
        da = dev(a)
        assert vc.lib().vc_f2sp_prove(s, da.data_ptr(), buf.data_ptr() + offset, None) == vc.VC_OK
        torch.cuda.synchronize()
    finally:
        vc.vc_f2sp_destroy(s)
    got = buf.cpu().numpy()
    assert (got[offset:offset + 16 * h].view(np.uint64) == want).all()
    assert (got[:offset] == 0x5A).all() and (got[offset + 16 * h:] == 0x5A).all()
