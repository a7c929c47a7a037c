"""The allocation-free time sort's two ways, buckets and radix passes, at the
sizes and spreads where they meet: bucket and tile edges, ranges of fewer values
than buckets, keys that crowd one bucket, the ends of the key range, output in
the input's place, and a captured call."""
import ctypes as C

import numpy as np
import pytest

import workloads as W  # noqa: F401  (the tests' path)

pytestmark = pytest.mark.gpu
MAX = 1 << 20


@pytest.fixture(scope="module")
def G():
    from paper_2603_07327_gb300 import build as B
    B.build()
    import paper_2603_07327_gb300 as G
    G.load()
    return G


def call(G, torch, d_in, d_out, d_perm, stream):
    code = G.load().gpet_sort_times_noalloc(C.c_void_p(d_in.data_ptr()), d_in.numel(), C.c_void_p(d_out.data_ptr()),
                                            C.c_void_p(d_perm.data_ptr()), C.c_void_p(stream.cuda_stream))
    assert code == 0, G.load().gpet_last_error().decode()


def keys_of(rng, spread, n):
    u = lambda bits: rng.integers(0, 1 << bits, n, dtype=np.uint64)
    if spread == "even":
        return u(46)
    if spread == "offset":                    # a short range far from zero, across a power of two
        return u(34) + np.uint64((1 << 60) - (1 << 33))
    if spread == "ends":                      # both ends of the 64-bit range
        k = u(63) * np.uint64(2)
        k[rng.integers(0, n)] = np.uint64(2**64 - 1)
        k[rng.integers(0, n)] = np.uint64(0)
        return k
    if spread == "few":                       # fewer values than buckets
        return u(9)
    if spread == "equal":
        return np.full(n, 12345, np.uint64)
    if spread == "rising":
        return np.arange(n, dtype=np.uint64) * np.uint64(977)
    if spread == "crowded":                   # most keys in one bucket, some far away
        k = u(20)
        k[:: 50] = rng.integers(0, 1 << 62, len(k[:: 50]), dtype=np.uint64)
        return k
    return np.floor(rng.exponential(1.0, n) * 2.0**40).astype(np.uint64)   # "decay"


@pytest.mark.parametrize("spread", ["even", "offset", "ends", "few", "equal", "rising", "crowded", "decay"])
@pytest.mark.parametrize("n", [1, 31, 64, 65, 513, 4095, 4097, 152 * 1024 + 1, 300_007, MAX])
def test_spreads(G, spread, n):
    torch = pytest.importorskip("torch")
    k = keys_of(np.random.default_rng(n), spread, n)
    d_in = torch.from_numpy(k.view(np.int64)).cuda()
    d_out, d_perm = torch.full_like(d_in, -1), torch.full((n,), -1, dtype=torch.int32, device="cuda")
    st = torch.cuda.current_stream()
    want = np.argsort(k, kind="stable")
    for out in (d_out, d_in):                 # apart, then in place
        call(G, torch, d_in, out, d_perm, st)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().view(np.uint64), k[want])
        assert np.array_equal(d_perm.cpu().numpy(), want.astype(np.int32))


def test_captured(G):
    """A captured call sorts what its buffers hold at each replay, by either way."""
    torch = pytest.importorskip("torch")
    n = 70_001
    d_in = torch.zeros(n, dtype=torch.int64, device="cuda")
    d_out, d_perm = torch.empty_like(d_in), torch.empty(n, dtype=torch.int32, device="cuda")
    call(G, torch, d_in, d_out, d_perm, torch.cuda.current_stream())   # the device's set-up
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(G, torch, d_in, d_out, d_perm, torch.cuda.current_stream())
    for spread in ("even", "crowded", "even"):
        k = keys_of(np.random.default_rng(5), spread, n)
        d_in.copy_(torch.from_numpy(k.view(np.int64)))
        g.replay()
        torch.cuda.synchronize()
        want = np.argsort(k, kind="stable")
        assert np.array_equal(d_out.cpu().numpy().view(np.uint64), k[want])
        assert np.array_equal(d_perm.cpu().numpy(), want.astype(np.int32))
