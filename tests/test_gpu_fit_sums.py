"""The sums of m3e_fit_grad keep their accuracy however many candidates a thread adds: n copies of
one candidate give n times its chi2 and gradient.  (The rounding errors of a plain FP32 sum of
equal terms do not average out: 64 additions of one value are off by up to 2e-6.)"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = np.float32
N = 10_000_000


def _plain(v, n):
    s = F(0)
    for _ in range(n):
        s = F(s + v)
    return float(s)


@pytest.mark.parametrize("grad", [False, True])
def test_copies_of_a_candidate_add_up(cfg, grad):
    from paper_2206_11535_gb300 import m3e
    d = gen.workload("c4", n_frames=100)
    hits, off = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    truth = O.nominal_params()
    truth[:24] = d["truth_align"].reshape(-1)
    p = torch.tensor(np.asarray(truth), dtype=torch.float32, device="cuda")
    with m3e.Context(cfg, 0) as c:
        rec = {k: v.cpu().numpy() for k, v in c.select_frames_debug(hits, off).items()}
        cand = torch.from_numpy(m3e.kept_candidates(rec, d["off"])).cuda()
        chi2 = c.fit_chi2(hits, off, cand, p).cpu().numpy()
        # the candidate whose sum a plain chain of about the length of a thread's share changes most
        chain = N // (132 * 8 * 128)
        worst = int(np.argmax([abs(_plain(v, chain) / (chain * float(v)) - 1) for v in chi2]))
        assert abs(_plain(chi2[worst], chain) / (chain * float(chi2[worst])) - 1) > 5e-7
        one = cand[worst:worst + 1]
        s1, g1 = c.fit_grad(hits, off, one, p)
        s, g = c.fit_grad(hits, off, one.expand(N, 4).contiguous(), p, grad=grad)
        assert c.fit_valid_count() == N
    # the sum is rounded to FP32 once, and so is the single candidate's it is compared with
    ulp = 2.0 ** -23
    assert abs(float(s) / N / float(s1) - 1) <= ulp
    if grad:
        a, b = g.double().cpu().numpy() / N, g1.double().cpu().numpy()
        assert (np.abs(a - b) <= ulp * np.abs(b)).all(), (a, b)
