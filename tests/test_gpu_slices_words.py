"""The sliced MLP kernel on device words that earlier launches have left, launched by itself."""
import pytest
import torch

from paper_2608_22643_b200 import binding as nb
from tests import internals

pytestmark = pytest.mark.gpu


class Words:
    """A small stack whose rows are resident, and the words a launch meets its other blocks in."""

    def __init__(self, lib, D, C, k, L, seed=3):
        self.lib, self.shape = lib, (D, C, k, L)
        self.sms = torch.cuda.get_device_properties(0).multi_processor_count
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.rows = [(torch.randn(L, C, D, generator=g, device="cuda") * 0.02).to(torch.bfloat16) for _ in range(3)]
        self.slots = torch.stack([torch.randperm(C, generator=g, device="cuda") for _ in range(L)]).to(torch.int32)
        self.counters = torch.zeros(L, nb.NP_N_COUNTERS, dtype=torch.int32, device="cuda")
        self.counters[:, nb.NP_CNT_ACTIVE] = k
        self.x = torch.randn(D, generator=g, device="cuda").to(torch.bfloat16)
        self.acc = torch.zeros(5, 16 * D, device="cuda")       # x and the fp32 accumulators
        self.out = torch.empty(D, device="cuda")
        n = (internals.C.c_ulonglong * 3)()
        lib.t_slices_words(D, C, k, self.sms, n)
        self.zfix, self.xch = (torch.zeros(v, dtype=torch.int64, device="cuda") for v in (n[0], n[2]))
        self.bars = torch.zeros(n[1], dtype=torch.int32, device="cuda")
        self.status = torch.zeros(4, dtype=torch.int32, device="cuda")
        self.base = internals.uints(0, 0, 0)

    def run(self):
        t = [*self.rows, self.slots, self.counters, self.x, *self.acc, self.out, self.status, self.zfix, self.bars, self.xch]
        stream = torch.cuda.current_stream().cuda_stream
        rc = self.lib.t_slices(*self.shape, self.sms, internals.pointers(*[v.data_ptr() for v in t]), self.base,
                               internals.C.c_void_p(stream))
        torch.cuda.synchronize()
        assert rc == 0 and self.base[2] == 1
        return self.out.clone(), int(self.status[0])

    def reference(self):
        D, _, k, L = self.shape
        x = self.x.double()
        for l in range(L):
            s = self.slots[l, :k].long()
            n = x / torch.sqrt((x * x).mean() + 1e-6)
            g, u = (self.rows[i][l][s].double() @ n for i in (0, 1))
            x = x + (g / (1 + torch.exp(-g)) * u) @ self.rows[2][l][s].double()
        return x


@pytest.fixture(scope="module")
def lib():
    return internals.load()


@pytest.mark.parametrize("D", [256, 2048])
@pytest.mark.parametrize("words", ["zero", "ones", "random"])
def test_sums_left_by_earlier_launches(lib, D, words):
    """The counted sums only grow and wrap: a launch starts from whatever they hold, all bits set among it."""
    w = Words(lib, D, 512, 60, 3)
    want, status = w.run()
    assert status == 0
    assert ((want.double() - w.reference()).norm() / w.reference().norm()).item() < 1e-5    # fp32 sums: 1e-6
    if words == "ones":     # the four words of a lane's two columns differ in every bit
        w.zfix.zero_()
        w.zfix[:D:2] = -1
    elif words == "random":
        w.zfix.random_(-2 ** 62, 2 ** 62).mul_(2)
    got, status = w.run()
    assert status == 0
    assert torch.equal(got.view(torch.int32), want.view(torch.int32))
