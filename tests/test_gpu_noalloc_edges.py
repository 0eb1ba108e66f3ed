"""qieo_generation_noalloc at the edges of its kernels: rows that end inside a lane's 8 genes
or inside a tile of 256, rows and buffers that start at any even (angle indices) or odd
(alleles) address, item sums that need 64 bits, and populations with more rows than warps.

Every output is compared with the CPU oracle. All results are whole numbers: the tolerance
is zero."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_30862_gb300 import qieo as Q
from paper_2609_30862_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Q.load()
    return torch


def _problem(ng, items):
    if items == "byte":
        return W.knapsack(ng, ng + 3)
    r = np.random.RandomState(ng)
    if items == "word":          # 16-bit items at the limit of the 32-bit sums
        w = r.randint(1, 65536, ng)
        w[::3] = 65535
        v = np.full(ng, 65535)
    else:                        # 32-bit items, values of both signs
        w = r.randint(0, 2**31 - 1, ng)
        v = r.randint(-2**31 + 1, 2**31 - 1, ng)
    return W.custom_problem(w, v, int(w.astype(np.int64).sum()) // 2)


@pytest.mark.parametrize("ng,np_,rule,D,items,koff,xoff", [
    (1, 3, 0, 4, "byte", 0, 0), (5, 40, 1, 8, "long", 1, 3), (7, 9, 0, 100, "word", 3, 1),
    (8, 33, 1, 100, "byte", 0, 5), (9, 64, 0, 12, "long", 7, 7), (255, 21, 0, 100, "word", 0, 0),
    (256, 20, 1, 100, "byte", 5, 2), (257, 19, 0, 4, "long", 0, 0), (263, 35, 1, 1200, "byte", 2, 4),
    (511, 12, 0, 100, "long", 1, 1), (2049, 700, 0, 100, "byte", 0, 0), (1003, 2500, 1, 8, "word", 6, 6),
])
def test_noalloc_edges(torch_cuda, ng, np_, rule, D, items, koff, xoff):
    torch = torch_cuda
    prob = _problem(ng, items)
    dev = torch.device("cuda", 0)
    n = np_ * ng
    d_w, d_v = torch.from_numpy(prob.weights).to(dev), torch.from_numpy(prob.values).to(dev)
    # guard elements on both sides of the shifted buffers: nothing outside may change
    kb = torch.full((n + 32,), 77, dtype=torch.int16, device=dev)
    xb = torch.full((n + 32,), 55, dtype=torch.uint8, device=dev)
    kb[8 + koff:8 + koff + n] = 0
    d_f = torch.zeros(np_, dtype=torch.int64, device=dev)
    d_e = torch.full((1,), -1, dtype=torch.int32, device=dev)
    p = Q.qieo_default_params()
    p.np, p.seed, p.instance_id, p.rotate_rule, p.dtheta_den, p.penalty_lambda = np_, 5, 2, rule, D, 2
    p.stream = torch.cuda.current_stream(dev).cuda_stream
    st = None
    for t in range(4):
        Q.qieo_generation_noalloc(d_w.data_ptr(), d_v.data_ptr(), ng, prob.capacity, p, t,
                                  kb.data_ptr() + 2 * (8 + koff), xb.data_ptr() + 8 + xoff,
                                  d_f.data_ptr(), d_e.data_ptr())
        st = O.run(prob, np_, 1, seed=5, inst=2, D=D, lam=2, rule=rule, state=st)
        torch.cuda.synchronize()
        k, x = kb.cpu().numpy(), xb.cpu().numpy()
        assert np.array_equal(x[8 + xoff:8 + xoff + n].reshape(np_, ng), st.x), t
        assert np.array_equal(d_f.cpu().numpy(), st.f), t
        assert int(d_e.cpu()[0]) == int(st.hist_e[-1]), t
        assert np.array_equal(k[8 + koff:8 + koff + n].reshape(np_, ng), st.k), t
        assert (k[:8 + koff] == 77).all() and (k[8 + koff + n:] == 77).all(), t
        assert (x[:8 + xoff] == 55).all() and (x[8 + xoff + n:] == 55).all(), t
