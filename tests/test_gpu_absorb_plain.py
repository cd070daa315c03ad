"""tn_absorb and tn_absorb_dot in FP32 on whole numbers, whose products FP32 holds
exactly: the absorption and, with every product compensated, the dot are exact."""
import pytest

from paper_1908_08553_gb300 import tn

pytestmark = pytest.mark.gpu


def _whole(g, shape, most):
    """Positive, so that four products no longer fit FP32's 24 bits."""
    import torch
    return torch.randint(most // 2, most + 1, shape, generator=g).float()


def _inputs(K, N, P, S, seed):
    """Outputs of at most 3600, products with adj below 2^24."""
    import torch
    g = torch.Generator().manual_seed(seed)
    most = int((3600 / K) ** 0.5)
    return _whole(g, (P, K, S), most), _whole(g, (K, N), most), _whole(g, (P, N, S), 4095)


# along s (S a multiple of 4), along p (S = 1, P a multiple of 4): the last 4 positions of a
# tile of 512, one past it, and a single group
@pytest.mark.parametrize("K,N", [(1, 1), (1, 16), (4, 1), (4, 16), (16, 1), (16, 4), (16, 16)])
@pytest.mark.parametrize("P,S", [(1, 4), (3, 12), (64, 32), (129, 16), (4, 1), (512, 1), (516, 1), (2048, 1)])
def test_whole_numbers_are_exact(K, N, P, S):
    import torch
    x, E, adj = _inputs(K, N, P, S, 1000 * K + 10 * N + P + S)
    y = torch.einsum("pks,kn->pns", x.double(), E.double())
    dot = float((y * adj.double()).sum())
    xd, Ed, ad = x.cuda(), E.cuda(), adj.cuda()
    out, res = torch.empty((P, N, S), device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    tn.tn_absorb(1, xd, Ed, out, P, K, N, S, st)
    tn.tn_absorb_dot(1, xd, Ed, ad, P, K, N, S, res, st)
    torch.cuda.synchronize()
    assert torch.equal(out.cpu().double(), y)
    assert float(res[0]) == dot


# pointers off a 16-byte boundary: the kernel of one position per thread; its sum of N
# products leaves rounded to FP32, 2^-24 of at most N 2^24 a position
@pytest.mark.parametrize("K,N,P,S", [(16, 16, 8, 64), (16, 4, 512, 1), (4, 16, 3, 12)])
def test_pointers_off_a_16_byte_boundary(K, N, P, S):
    import torch
    x, E, adj = _inputs(K, N, P, S, 7 + K + N)
    y = torch.einsum("pks,kn->pns", x.double(), E.double())

    def off(t):
        b = torch.empty(t.numel() + 1, device="cuda")
        b[1:] = t.flatten().cuda()
        return b[1:]

    xd, ad, Ed, out = off(x), off(adj), E.cuda(), off(torch.zeros(P, N, S))
    res = torch.zeros(1, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    tn.tn_absorb(1, xd, Ed, out, P, K, N, S, st)
    tn.tn_absorb_dot(1, xd, Ed, ad, P, K, N, S, res, st)
    torch.cuda.synchronize()
    assert torch.equal(out.cpu().double().reshape(P, N, S), y)
    assert abs(float(res[0]) - float((y * adj.double()).sum())) <= P * S * N
