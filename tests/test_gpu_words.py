"""The resident MLP kernels on device words that earlier launches have left, launched by themselves."""
import pytest
import torch

from paper_2608_22643_b200 import binding as nb
from tests import internals

pytestmark = pytest.mark.gpu


TIMEOUT = 8     # the status bit of a wait that ran out


class Words:
    """A small stack whose rows are resident, and the words a launch meets its other blocks in."""

    def __init__(self, lib, D, C, k, L, B=1, seed=3):
        self.lib, self.shape, self.B = lib, (D, C, k, L), B
        self.sms = torch.cuda.get_device_properties(0).multi_processor_count
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.rows = [(torch.randn(L, C, D, generator=g, device="cuda") * 0.02).to(torch.bfloat16) for _ in range(3)]
        self.slots = torch.stack([torch.randperm(C, generator=g, device="cuda") for _ in range(L)]).to(torch.int32)
        self.counters = torch.zeros(L, nb.NP_N_COUNTERS, dtype=torch.int32, device="cuda")
        self.counters[:, nb.NP_CNT_ACTIVE] = k
        self.x = torch.randn(B, D, generator=g, device="cuda").to(torch.bfloat16)
        self.acc = torch.zeros(5, 16 * D, device="cuda")       # x and, for one sequence, the fp32 accumulators
        self.out = torch.empty(B, D, device="cuda")
        n = (internals.C.c_ulonglong * 3)()
        if B == 1:
            lib.t_slices_words(D, C, k, self.sms, n)
            kinds = (torch.int64, torch.int32, torch.int64)     # counted sums, arrivals, exchange words
        else:
            lib.t_batch_words(self.sms, n)
            kinds = (torch.int32, torch.int64)                  # arrivals, exchange words
        self.words = [torch.zeros(v, dtype=t, device="cuda") for v, t in zip(n, kinds)]
        self.status = torch.zeros(4, dtype=torch.int32, device="cuda")
        self.base = internals.uints(0, 0, 0)

    def clear(self):
        for w in [*self.words, self.status]:
            w.zero_()
        self.base = internals.uints(0, 0, 0)

    def run(self):
        acc = self.acc if self.B == 1 else self.acc[:1]
        t = [*self.rows, self.slots, self.counters, self.x, *acc, self.out, self.status, *self.words]
        ptr = internals.pointers(*[v.data_ptr() for v in t])
        stream = internals.C.c_void_p(torch.cuda.current_stream().cuda_stream)
        if self.B == 1:
            rc = self.lib.t_slices(*self.shape, self.sms, ptr, self.base, stream)
        else:
            rc = self.lib.t_batch(*self.shape, self.B, self.sms, ptr, self.base, stream)
        torch.cuda.synchronize()
        assert rc == 0
        return self.out.clone(), int(self.status[0])

    def error(self, got):
        D, _, k, L = self.shape
        x = self.x.double()
        for l in range(L):
            s = self.slots[l, :k].long()
            n = x / torch.sqrt((x * x).mean(dim=1, keepdim=True) + 1e-6)
            g, u = (n @ self.rows[i][l][s].double().T for i in (0, 1))
            x = x + (g / (1 + torch.exp(-g)) * u) @ self.rows[2][l][s].double()
        return ((got.double() - x).norm() / x.norm()).item()


@pytest.fixture(scope="module")
def lib():
    return internals.load()


@pytest.mark.parametrize("D", [256, 2048])
@pytest.mark.parametrize("words", ["zero", "ones", "random"])
def test_sums_left_by_earlier_launches(lib, D, words):
    """The counted sums only grow and wrap: a launch starts from whatever they hold, all bits set among it."""
    w = Words(lib, D, 512, 60, 3)
    want, status = w.run()
    assert status == 0 and w.error(want) < 1e-5    # fp32 sums: 1e-6
    zfix = w.words[0]
    if words == "ones":     # the four words of a lane's two columns differ in every bit
        zfix.zero_()
        zfix[:D:2] = -1
    elif words == "random":
        zfix.random_(-2 ** 62, 2 ** 62).mul_(2)
    got, status = w.run()
    assert status == 0
    assert torch.equal(got.view(torch.int32), want.view(torch.int32))


@pytest.mark.parametrize("B,D", [(1, 256), (1, 4096), (1, 8192), (4, 256), (16, 2048)])
def test_a_wait_that_runs_out(lib, B, D):
    """The launch waits for an arrival that nobody makes: it says so, ends, and the words cleared it runs as before."""
    w = Words(lib, D, 1024, 37 * 20, 4, B)      # more rows than a block's ring holds: copies are under way at the end
    want, status = w.run()
    assert status == 0 and w.error(want) < 1e-5
    w.base[0] += 1                              # one arrival more than the blocks make
    _, status = w.run()
    assert status == TIMEOUT
    w.clear()
    got, status = w.run()
    assert status == 0 and w.error(got) < 1e-5


# A multiplication that adds to a long chain truncates at every step.  Mean of four inputs with one chain per tile and the warps'
# sums added one after the other 3.06e-7, 7.41e-7, 8.53e-7; two chains and sums in pairs 2.74e-7, 5.84e-7, 6.67e-7.  The same
# inputs give the same bits, so a limit between them tells them apart.
@pytest.mark.parametrize("D,k,most", [(2384, 600, 2.9e-7), (4112, 1101, 6.6e-7), (5120, 1382, 7.6e-7)])
def test_error_of_the_sums(lib, D, k, most):
    """20 layers against 64-bit sums."""
    errors = []
    for seed in range(4):
        w = Words(lib, D, k + 100, k, 20, seed=seed)
        got, status = w.run()
        assert status == 0
        errors.append(w.error(got))
    assert sum(errors) / 4 < most


@pytest.mark.parametrize("B,D,rows", [(1, 4096, 37 * 64), (1, 8192, 37 * 64), (3, 4096, 37 * 80), (16, 2048, 37 * 80)])
def test_a_wait_that_runs_out_laps_before_the_end(lib, B, D, rows):
    """The same with several laps of a block's ring left when the wait runs out: none of its slots is filled any more."""
    w = Words(lib, D, 3072, rows, 4, B)
    want, status = w.run()
    assert status == 0 and w.error(want) < 1e-5
    w.base[0] += 1
    _, status = w.run()
    assert status == TIMEOUT
    w.clear()
    got, status = w.run()
    assert status == 0 and w.error(got) < 1e-5


@pytest.mark.parametrize("D,k", [(1024, 1500), (4096, 1100)])
def test_a_wait_that_runs_out_in_a_cluster(lib, D, k):
    """The same for the kernel that deals whole rows to the blocks of clusters."""
    L = 7                                           # several laps of its ring
    w = Words(lib, D, k + 100, k, L)
    acc = torch.zeros(int(lib.t_rows_words(D)), device="cuda")
    cnt = torch.zeros(4, dtype=torch.int32, device="cuda")
    t = [*w.rows, w.slots, w.counters, w.x, *w.acc, w.out, w.status, acc, cnt]

    def run():
        stream = internals.C.c_void_p(torch.cuda.current_stream().cuda_stream)
        rc = lib.t_rows(*w.shape, w.sms, internals.pointers(*[v.data_ptr() for v in t]), w.base, stream)
        torch.cuda.synchronize()
        assert rc == 0
        return w.acc[(L - 1) & 1, :D].clone().view(1, D), int(w.status[0])

    want, status = run()
    assert status == 0 and w.error(want) < 1e-5
    w.base[0] += 1
    _, status = run()
    assert status == TIMEOUT
    for v in (acc, cnt, w.acc):
        v.zero_()
    w.clear()
    got, status = run()
    assert status == 0 and w.error(got) < 1e-5
