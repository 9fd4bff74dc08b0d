"""Products of at most 128 columns: one launch that expands the packed weights as it
multiplies, the reduction of ten stages of 64 indices or more split over a cluster
where the SMs hold it.  Every output against the fp64 oracle at the tolerance of all
products (1e-5 of sum |w||x|), with the output stage's bf16 rounding where it applies;
that the launch ran is shown by the workspace, which it leaves as it is."""
import numpy as np
import pytest
import torch

import oracle
import paper_1910_11971_gb300 as cci
from paper_1910_11971_gb300 import workloads as wl
from parity_util import TOL, assert_within_tol, f64, oracle_reference

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


@pytest.fixture(scope="module")
def dev():
    return torch.device("cuda:0")


# columns at the edges of the MMA's N (16, 32, 64, 128); reductions of one chunk and
# less, at both edges of the rule (7 stages, 10), with a ragged last stage, and deep
# enough for 2, 4 and 8 parts of unequal length; channels below, at and past a tile of
# 128, at the last tile count that is split (76) and past it, and more tiles than SMs;
# every K, G 4 to 32
CASES = [
    (1, 8, 8, 8, 2), (7, 16, 1360, 8, 1), (33, 72, 24, 4, 2), (128, 448, 224, 32, 8), (100, 584, 136, 8, 4),
    (16, 640, 96, 16, 8), (1, 1024, 64, 4, 1), (16, 1032, 72, 8, 2), (17, 1536, 1000, 8, 4), (32, 2048, 128, 16, 8),
    (33, 1096, 136, 4, 2), (64, 4096, 256, 32, 4), (65, 2056, 160, 32, 1), (100, 2048, 1000, 8, 1),
    (127, 1160, 96, 16, 2), (128, 3000, 264, 8, 2), (5, 1024, 20, 4, 1), (128, 4096, 4096, 16, 4),
    (40, 1024, 4608, 8, 2), (3, 640, 9728, 8, 2), (128, 640, 9736, 8, 4), (5, 1032, 19584, 8, 2),
]


@pytest.mark.parametrize("N,Cin,Cout,G,K", CASES)
def test_narrow_product(dev, N, Cin, Cout, G, K):
    X, W = wl.random_small(N + Cin + Cout, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    st = cci.new_status(dev)
    ws = torch.full((Cout * Cin * 2,), 0xA5, dtype=torch.uint8, device=dev)
    Y = cci.linear(X.to(dev), v, i, Cout, G, K, status=st, workspace=ws)
    assert cci.read_status(st) == 0
    assert bool((ws == 0xA5).all())  # the one launch ran
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.linear(f64(X), Wd, mask)
    assert_within_tol(f64(Y), Yo, S, f"narrow product {N} x {Cin} -> {Cout}")


# (N, Cin, G, K): one column too many, eight and nine stages (with ragged ends), K = 16
@pytest.mark.parametrize("N,Cin,G,K", [(129, 1024, 8, 2), (1, 456, 8, 2), (64, 512, 8, 1), (128, 512, 16, 8),
                                       (100, 576, 4, 2), (128, 576, 32, 8), (16, 1024, 32, 16)])
def test_past_the_rule_the_workspace_family_runs(dev, N, Cin, G, K):
    Cout = 224
    X, W = wl.random_small(N + Cin, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    ws = torch.full((Cout * Cin * 2,), 0xA5, dtype=torch.uint8, device=dev)
    Y = cci.linear(X.to(dev), v, i, Cout, G, K, workspace=ws)
    _, _, Wd, mask = oracle_reference(W, G, K)
    assert (f64(ws.view(BF16)).reshape(Cout, Cin) == Wd).all()
    Yo, S = oracle.linear(f64(X), Wd, mask)
    assert_within_tol(f64(Y), Yo, S, f"workspace product {N} x {Cin} -> {Cout}")


def test_infinite_and_nan_activations(dev):
    """A pruned weight times an infinity or a NaN is NaN, as in the dense product of
    the workspace family; the other columns are untouched by it."""
    N, Cin, Cout, G, K = 33, 1096, 136, 8, 2
    X, W = wl.random_small(6, "bf16", N, Cin, Cout)
    X[3, 700] = float("inf")
    X[20, 1095] = float("-inf")
    X[32, 0] = float("nan")
    v, i = cci.pack(W.to(dev), G, K)
    Y = f64(cci.linear(X.to(dev), v, i, Cout, G, K))
    Yw = f64(cci.linear(X.to(dev), v, i, Cout, G, K, algo=cci.ALGO_DENSE_TC_WS))
    assert (np.isnan(Y) == np.isnan(Yw)).all() and np.isnan(Y[[3, 20, 32]]).any(axis=1).all()
    assert (np.isposinf(Y) == np.isposinf(Yw)).all() and (np.isneginf(Y) == np.isneginf(Yw)).all()
    assert np.isinf(Y[[3, 20]]).any()
    rest = np.setdiff1d(np.arange(N), [3, 20, 32])
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.linear(f64(X[rest]), Wd, mask)
    assert_within_tol(Y[rest], Yo, S, "finite columns")


@pytest.mark.parametrize("N,Cin,Cout,G,K", [(16, 1024, 136, 8, 2), (100, 2048, 1000, 8, 4), (3, 4096, 96, 32, 8)])
@pytest.mark.parametrize("bf16_out", [False, True])
def test_narrow_product_output_stage(dev, N, Cin, Cout, G, K, bf16_out):
    X, W = wl.random_small(7 + N, "bf16", N, Cin, Cout)
    bias = torch.linspace(-2.0, 2.0, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    Y = cci.linear_fused(X.to(dev), v, i, Cout, G, K, bias=bias.to(dev), relu=True,
                         out_dtype=BF16 if bf16_out else torch.float32)
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.linear(f64(X), Wd, mask)
    b = f64(bias)
    ref = np.maximum(Yo + b, 0.0)
    lim = TOL * (S + np.abs(b)) + (2.0 ** -8 * np.abs(ref) if bf16_out else 0.0)
    assert (np.abs(f64(Y) - ref) <= lim).all()


def test_narrow_product_reports_bad_index_sets(dev):
    """An index >= G, a repeated and an unordered index, each alone in the last
    group and the last reduction index, are reported."""
    N, Cin, Cout, G, K = 8, 1032, 264, 8, 4
    X, W = wl.random_small(3, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    for bad in ([0, 1, 2, G], [0, 1, 1, 2], [0, 2, 1, 3], [255, 1, 2, 3]):
        j = i.clone()
        j[-1, -1] = torch.tensor(bad, dtype=torch.uint8)
        st = cci.new_status(dev)
        cci.linear(X.to(dev), v, j, Cout, G, K, status=st)
        assert cci.read_status(st) == 10, bad


def bad_sets(G, K):
    """Index sets with one fault each: two neighbouring slots equal or swapped, for every
    pair of slots, and a last index at and above G."""
    good = list(range(K))
    sets = [good[:-1] + [G], good[:-1] + [255]]
    for s in range(K - 1):
        sets += [good[:s + 1] + [s] + good[s + 2:], good[:s] + [s + 1, s] + good[s + 2:]]
    return sets


# few columns (the one launch); the decompression and the fused family, whatever the columns
@pytest.mark.parametrize("G,K", [(4, 1), (32, 1), (4, 2), (32, 2), (8, 4), (32, 4), (16, 8), (32, 8)])
@pytest.mark.parametrize("N,algo", [(8, cci.ALGO_AUTO), (8, cci.ALGO_DENSE_TC_WS), (200, cci.ALGO_DENSE_TC_WS),
                                    (200, cci.ALGO_DENSE_TC)], ids=["few", "ws8", "ws200", "fused"])
def test_bad_index_sets_are_reported(dev, N, algo, G, K):
    """Each fault alone, in the first and the last set, and at a set that starts at
    another byte of its word, is reported; the untouched sets are not."""
    Cin, Cout = 1040, 96
    X, W = wl.random_small(3, "bf16", N, Cin, Cout)
    X = X.to(dev)
    v, i = cci.pack(W.to(dev), G, K)

    def status_of(j):
        st = cci.new_status(dev)
        cci.linear(X, v, j, Cout, G, K, status=st, algo=algo)
        return cci.read_status(st)

    assert status_of(i) == 0
    assert status_of(torch.arange(G - K, G, dtype=torch.uint8, device=dev).expand_as(i).contiguous()) == 0
    for bad in bad_sets(G, K):
        for at in ((0, 0), (i.shape[0] // 2, 5), (-1, -1)):
            j = i.clone()
            j[at] = torch.tensor(bad, dtype=torch.uint8)
            assert status_of(j) == 10, (bad, at)


@pytest.mark.parametrize("N,chunk", [(100, 32), (300, 100)])
def test_host_chunks_keep_the_bits_of_the_whole(dev, N, chunk):
    """A host-buffer product cut into chunks of few columns equals the whole
    product bit for bit: below and above the rule's 128 columns."""
    Cin, Cout, G, K = 2048, 264, 8, 2
    X, W = wl.random_small(11, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    Y = cci.linear(X.to(dev), v, i, Cout, G, K).cpu()
    Yh = cci.linear_host(X.pin_memory(), v, i, Cout, G, K, chunk=chunk)
    torch.cuda.synchronize()
    assert torch.equal(Y.view(torch.int32), Yh.view(torch.int32))


@pytest.mark.parametrize("N,Cin,Cout,G,K", [(1, 256, 136, 8, 2), (100, 640, 96, 16, 8), (128, 1024, 64, 4, 1)])
def test_workspace_family_by_name_leaves_the_dense_weights(dev, N, Cin, Cout, G, K):
    """Asked for by name, the workspace family decompresses into the workspace whatever
    the columns and gives a column the bits it has in a call of many columns; AUTO
    leaves a workspace as it is there, which also shows that its one launch ran."""
    X, W = wl.random_small(5 + N, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    many = torch.cat([X, X, torch.randn((300, Cin)).to(BF16)]).to(dev)
    ws = torch.full((Cout * Cin * 2,), 0xA5, dtype=torch.uint8, device=dev)
    args = (v, i, Cout, G, K)
    Y = cci.linear(X.to(dev), *args, algo=cci.ALGO_AUTO, workspace=ws)
    assert bool((ws == 0xA5).all())
    Yw = cci.linear(X.to(dev), *args, algo=cci.ALGO_DENSE_TC_WS, workspace=ws)
    _, _, Wd, mask = oracle_reference(W, G, K)
    assert (f64(ws.view(BF16)).reshape(Cout, Cin) == Wd).all()
    Ym = cci.linear(many, *args, algo=cci.ALGO_DENSE_TC_WS)
    assert torch.equal(Yw.view(torch.int32), Ym[:N].view(torch.int32))
    Yo, S = oracle.linear(f64(X), Wd, mask)
    assert_within_tol(f64(Y), Yo, S, "AUTO")
    assert_within_tol(f64(Yw), Yo, S, "workspace family by name")
    Ys = torch.empty_like(Yw)  # the static-array entry is the workspace family by name
    Xd = X.to(dev)
    assert cci.lib().cci_linear_dense_tc_static(Xd.data_ptr(), cci.BF16, N, Cin, v.data_ptr(), i.data_ptr(), Cout, G, K,
                                                Ys.data_ptr(), None, cci._stream(dev)) == 0
    assert torch.equal(Ys.view(torch.int32), Yw.view(torch.int32))


def plain_call(X, v, i, Cout, G, K, epilogue, workspace=None):
    """(status code, Y) of the C call without the binding's workspace: cci_linear_ws with
    AUTO, or cci_linear_fused without bias and ReLU."""
    Y = torch.zeros((X.shape[0], Cout), dtype=torch.float32, device=X.device)
    head = (X.data_ptr(), cci.BF16, X.shape[0], X.shape[1], v.data_ptr(), i.data_ptr(), Cout, G, K)
    ws = (None, 0) if workspace is None else (workspace.data_ptr(), workspace.numel())
    if epilogue:
        code = cci.lib().cci_linear_fused(*head, None, 0, cci.F32, Y.data_ptr(), None, *ws, cci._stream(X.device))
    else:
        code = cci.lib().cci_linear_ws(*head, Y.data_ptr(), None, cci.ALGO_AUTO, *ws, cci._stream(X.device))
    return code, Y


@pytest.mark.parametrize("N,Cin,Cout,G,K", [(8, 384, 40, 8, 2), (100, 2048, 144, 16, 8), (128, 1024, 264, 4, 1)])
def test_one_launch_without_a_workspace(dev, N, Cin, Cout, G, K):
    """Without a workspace the layer runs the same launch, with the same bits, through
    the plain entry point and the one with an output stage as with a workspace (which
    stays unwritten: the launch that reads none ran)."""
    X, W = wl.random_small(9 + N, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    Xd = X.to(dev)
    ws = torch.full((Cout * Cin * 2,), 0xA5, dtype=torch.uint8, device=dev)
    outs = [plain_call(Xd, v, i, Cout, G, K, ep, w) for ep in (False, True) for w in (ws, None)]
    assert [code for code, _ in outs] == [0] * 4
    assert bool((ws == 0xA5).all())
    for _, Y in outs[1:]:
        assert torch.equal(Y.view(torch.int32), outs[0][1].view(torch.int32))
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.linear(f64(X), Wd, mask)
    assert_within_tol(f64(outs[0][1]), Yo, S, "no workspace")


def test_layers_that_need_a_workspace_still_ask_for_it(dev):
    """R * K no multiple of 16: the fused family does not have the layer, so without a
    workspace the output stage is refused and AUTO runs on the CUDA cores."""
    N, Cin, Cout, G, K = 8, 1032, 72, 8, 1
    X, W = wl.random_small(2, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    assert plain_call(X.to(dev), v, i, Cout, G, K, True)[0] == 11
    code, Y = plain_call(X.to(dev), v, i, Cout, G, K, False)
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.linear(f64(X), Wd, mask)
    assert code == 0
    assert_within_tol(f64(Y), Yo, S, "AUTO without a workspace")


@pytest.mark.parametrize("captured", [False, True])
def test_launches_in_a_row_read_what_the_ones_before_wrote(dev, captured):
    """Each launch may be scheduled before the one ahead has ended: a chain of layers in
    one stream, called and as a CUDA graph, equals the same layers with a wait after
    each, bit for bit."""
    N, C, G, K, depth = 32, 1024, 8, 2, 40
    g = torch.Generator().manual_seed(4)
    X0 = torch.randn((N, C), generator=g).to(BF16).to(dev)
    packed = [cci.pack((torch.randn((C, C), generator=g) * (2.0 / C) ** 0.5).to(BF16).to(dev), G, K)
              for _ in range(3)]

    def chain(wait):
        x, outs = X0, []
        for n in range(depth):
            v, i = packed[n % 3]
            x = cci.linear_fused(x, v, i, C, G, K, relu=n % 2 == 0, out_dtype=BF16)
            outs.append(x)
            if wait:
                torch.cuda.synchronize()
        return outs

    want = chain(True)
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            got = chain(False)
        graph.replay()
    else:
        got = chain(False)
    torch.cuda.synchronize()
    for n, (a, b) in enumerate(zip(got, want)):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), n
    assert bool(want[-1].isfinite().all()) and bool((want[-1] != 0).any())
