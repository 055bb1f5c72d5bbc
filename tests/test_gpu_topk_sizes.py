"""Selection at the column lengths where the top-k kernel changes form (scores per thread,
threads, keys in shared memory from 8193 scores, over a cluster of eight CTAs from 49153, and the
scan over global memory above 393216), on columns that start on and off the 16-byte grid, and the
output forms of ec_route: scores returned in place, to an array that the kernels cannot write
directly, and not at all. Exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import ecmoe as O
from paper_2604_01622_gb300 import ec_route
from paper_2604_01622_gb300.layer import ECMoELayer

pytestmark = pytest.mark.gpu


def _scores(rng, N, E, kind):
    if kind == "narrow":          # a softmax column: a spread of a few percent
        return (np.exp(0.03 * rng.standard_normal((N, E))) / E).astype(np.float32)
    if kind == "ties":            # few distinct values, the k-th one shared by many tokens
        return (np.round(rng.random((N, E)) * 6) / 8).astype(np.float32)
    s = rng.standard_normal((N, E)).astype(np.float32)   # both signs: offsets over 31 bits
    s[rng.random((N, E)) < 0.01] = np.float32(-0.0)
    s[0], s[N // 2] = np.float32(3e38), np.float32(-3e38)
    return s


@pytest.mark.parametrize("kind", ["narrow", "ties", "signed"])
@pytest.mark.parametrize("L", [1, 509, 512, 513, 2045, 2048, 2049, 4096, 8189, 8192, 8193, 16384,
                               16385, 32768, 32769, 49152, 49153, 131077, 393216, 393217])
def test_selection_at_every_kernel_form(L, kind):
    rng = np.random.default_rng(L)
    E, tail = 3, 6                # a second, short group; N = L + 6 moves columns off the grid
    for head in (0, 1):           # head = 1: an extra one-token group shifts the long one
        group_off = np.array([0, head, head + L, head + L + tail], np.int32)
        N = int(group_off[-1])
        k_g = np.array([head, max(1, L // 8), 2], np.int32)
        S = _scores(rng, N, E, kind)
        lay = ECMoELayer(N, 64, E, 64, group_off, k_g, dtype="f32")
        ST = torch.from_numpy(np.ascontiguousarray(S.T)).cuda()
        idx, gate, S_out = lay.route(S_in=ST)
        lay.check()
        ref_idx, _ = O.ec_select(S.astype(np.float64), group_off, k_g)
        assert np.array_equal(idx.cpu().numpy(), ref_idx)
        want = S.T[np.arange(E)[:, None], ref_idx]
        assert np.array_equal(gate.cpu().numpy().view(np.uint32), want.view(np.uint32))
        assert torch.equal(S_out.view(torch.int32), ST.view(torch.int32))
        lay.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_route_output_forms_agree(dtype):
    """Scores written by the kernels (aligned array), copied afterwards (array off the 16-byte
    grid, or overlapping the input scores), left in place and not asked for: the same values."""
    torch.manual_seed(3)
    N, d, E = 700, 64, 12
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    X = torch.randn(N, d, device="cuda").to(td)
    Wr = (torch.randn(d, E, device="cuda") / 8).to(td)
    lay = ECMoELayer(N, d, E, 64, np.array([0, 301, N]), np.array([40, 17]), dtype=dtype)
    st = torch.cuda.current_stream().cuda_stream
    M = lay.M
    idx0, gate0, S0 = lay.route(X, Wr)
    other = torch.empty(E * N + 1, device="cuda")[1:]

    def go(S_in, S_out):
        idx = torch.empty(E, M, dtype=torch.int32, device="cuda")
        gate = torch.empty(E, M, device="cuda")
        ec_route(lay.ctx, None if S_in is not None else X.data_ptr(),
                 None if S_in is not None else Wr.data_ptr(), None,
                 None if S_in is None else S_in.data_ptr(),
                 None if S_out is None else S_out.data_ptr(), idx.data_ptr(), gate.data_ptr(), st)
        lay.check()
        assert torch.equal(idx, idx0) and torch.equal(gate, gate0)
        if S_out is not None:
            assert torch.equal(S_out.reshape(-1)[:E * N], S0.reshape(-1))

    go(None, other)
    go(None, None)
    go(S0, None)
    go(S0, other)
    same = S0.clone()
    go(same, same)
    both = torch.empty(E * N + 4, device="cuda")
    both[4:] = S0.reshape(-1)
    go(both[4:], both[:E * N])        # S_out overlaps the second part of S_in
    Wg = (torch.randn(E, d, 64, device="cuda") / 8).to(td)
    Wd = (torch.randn(E, 64, d, device="cuda") / 8).to(td)
    _, idx, gate, S = lay.forward(X, Wr, None, Wg, Wg, Wd)
    assert torch.equal(idx, idx0) and torch.equal(gate, gate0) and torch.equal(S, S0)
