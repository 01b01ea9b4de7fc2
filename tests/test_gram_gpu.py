"""GPU parity of the exact-Gram reduction (TSQR_LEAF_GRAM) against the CPU oracle, at the sizes
where it can go wrong: the edges of its width classes, ragged row blocks, leading dimensions that
take the narrow copies, columns whose exponents rise while they are summed, and the matrices it
hands to the Householder reduction.  Bounds as in the FP64 parity tests: every entry within
c(m) kappa u ||R_oracle||_F, c(m) = max(50, 2 sqrt(m)), Gram residual <= 1e-13."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def T():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_4250_gb300 as T
    return T


def _check(oracle, R, At):
    A = oracle.from_torch_colmajor(At)
    R = R.cpu().numpy()
    Ro = oracle.householder_r(A, nthreads=16)
    assert np.all(np.tril(R, -1) == 0) and np.all(np.diag(R) >= 0)
    tol = max(50.0, 2.0 * np.sqrt(A.shape[0])) * oracle.kappa_from_r(Ro) * U * np.linalg.norm(Ro)
    np.testing.assert_allclose(R, Ro, rtol=0, atol=tol)
    assert oracle.gram_residual(A, R, nthreads=16) <= 1e-13


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 23, 24, 25, 31, 32])
@pytest.mark.parametrize("m,pad", [(1024, 0), (1087, 1), (70001, 0), (100003, 5)])
def test_widths_and_ragged_rows(oracle, T, n, m, pad):
    import torch
    At = workloads.gaussian(m, n, seed=600 + n)
    big = torch.full((n, m + pad), float("nan"), dtype=torch.float64)
    big[:, :m] = At
    R = T.tsqr_r(big.cuda().T[:m, :])
    assert T.last_plan().leaf == T.LEAF_GRAM and T.tsqr_last_launch_count() == 1
    _check(oracle, R, At)
    assert T.tsqr_get_device_status() == T.SUCCESS


@pytest.mark.parametrize("n", [5, 13, 30])
@pytest.mark.parametrize("kind", ["grow", "outlier", "constant", "scales", "kappa"])
def test_value_ranges(oracle, T, n, kind):
    """Columns that grow by 2^40 on the way (exponents rise often), one entry 2^30 above the
    rest in the middle, constant columns, columns of scales 2^-200 .. 2^200, kappa = 1e8."""
    import torch
    m = 150001
    At = workloads.gaussian(m, n, seed=650 + n)
    if kind == "grow":
        At *= torch.exp2(torch.arange(m, dtype=torch.float64) * (40.0 / m))
    elif kind == "outlier":
        At[:, m // 2] *= 2.0 ** 30
    elif kind == "constant":
        At[0] = 0.1
    elif kind == "scales":
        At *= torch.exp2(torch.linspace(-200, 200, n, dtype=torch.float64).round())[:, None]
    else:
        At = workloads.conditioned(m, n, 1e8, seed=n)
    R = T.tsqr_r(At.cuda().T)
    if kind == "scales":  # column j of R scales with column j of A, exactly
        s = torch.exp2(-torch.linspace(-200, 200, n, dtype=torch.float64).round())
        R, At = R.cpu() * s[None, :], At * s[:, None]
    _check(oracle, R, At)


@pytest.mark.parametrize("n", [6, 16, 32])
@pytest.mark.parametrize("kind", ["repeated", "zero", "zeros", "huge", "tiny", "nan", "inf"])
def test_what_the_householder_reduction_takes_over(oracle, T, n, kind):
    """Repeated and zero columns, entries whose squares leave FP64, NaN and Inf: the bytes and the
    status are those of the one Householder reduction with the same leaves."""
    import torch
    m = 60013
    At = workloads.gaussian(m, n, seed=700 + n)
    if kind == "repeated":
        At[n - 1] = At[1]
    elif kind == "zero":
        At[n // 2] = 0.0
    elif kind == "zeros":
        At.zero_()
    elif kind == "huge":
        At[2] *= 1e200
    elif kind == "tiny":
        At[2] *= 1e-200
    else:
        At[3, 12345] = float(kind)
    Ad = At.cuda().T
    T.tsqr_get_device_status()  # clears it
    R = T.tsqr_r(Ad)
    status = T.tsqr_get_device_status()
    p = T.last_plan()
    assert p.leaf == T.LEAF_GRAM
    ref = T.tsqr_r_ex(Ad, plan=T.make_plan("hybrid", tile_rows=p.tile_rows, ctas=p.ctas,
                                           warps=p.warps, arity=p.arity))
    assert T.last_plan().leaf == 0
    assert status == T.tsqr_get_device_status()
    assert torch.equal(torch.nan_to_num(R), torch.nan_to_num(ref))
    assert torch.equal(torch.isfinite(R), torch.isfinite(ref))
    if kind in ("repeated", "zero", "zeros"):
        A = oracle.from_torch_colmajor(At)
        if kind != "zeros":
            assert oracle.gram_residual(A, R.cpu().numpy(), nthreads=16) <= 1e-13
        assert status == T.SUCCESS


def test_capture_streams_and_plans(oracle, T):
    """A captured call replays on new data; two streams run side by side; the plan a call reports
    gives the same bytes; a plan that asks for the Gram where it does not serve is refused."""
    import torch
    m, n = 120000, 20
    A1, A2 = (workloads.gaussian(m, n, seed=s).cuda() for s in (1, 2))
    R1, R2 = T.tsqr_r(A1.T).clone(), T.tsqr_r(A2.T).clone()
    assert torch.equal(T.tsqr_r_ex(A1.T, plan=T.last_plan()), R1)
    buf, out = A1.clone(), T.empty_r(n, "cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        T.tsqr_r(buf.T, R=out)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        T.tsqr_r(buf.T, R=out, stream=s)
    buf.copy_(A2)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, R2)
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = []
    for k, st in enumerate(streams * 4):
        with torch.cuda.stream(st):
            outs.append((k, T.tsqr_r((A1 if k % 2 else A2).T)))
    torch.cuda.synchronize()
    for k, R in outs:
        assert torch.equal(R, R1 if k % 2 else R2)
    for bad in (T.make_plan("binary", tile_rows=256), T.make_plan("flat")):
        bad.leaf = T.LEAF_GRAM
        with pytest.raises(T.TsqrError) as e:
            T.tsqr_r_ex(A1.T, plan=bad)
        assert e.value.status == T.ERR_INVALID_ARG


@pytest.mark.parametrize("n", [33, 40, 41, 48, 49, 55, 56, 63, 64, 65, 72, 96, 97, 127, 128])
@pytest.mark.parametrize("m,pad", [(2048, 0), (30011, 3)])
def test_column_blocks(oracle, T, n, m, pad):
    """Past 32 columns the sums go by blocks of 32 columns, a block against itself or another."""
    import torch
    At = workloads.gaussian(m, n, seed=800 + n)
    At *= torch.exp2(torch.arange(m, dtype=torch.float64) * (6.0 / m))  # exponents rise
    big = torch.full((n, m + pad), float("nan"), dtype=torch.float64)
    big[:, :m] = At
    Ad = big.cuda().T[:m, :]
    R = T.tsqr_r(Ad)
    p = T.last_plan()
    assert (p.leaf, p.tree) == ((T.LEAF_GRAM, T.TREE_HYBRID) if n < 56 else (0, T.TREE_PANELS))
    _check(oracle, R, At)
    assert torch.equal(T.tsqr_r_ex(Ad, plan=p), R)


@pytest.mark.parametrize("n", [40, 100])
@pytest.mark.parametrize("kind", ["repeated", "zero", "nan", "kappa"])
def test_column_blocks_handed_over(oracle, T, n, kind):
    """What the Gram sum cannot serve runs the launches behind it: the Householder reduction's
    bytes (its own plan, or panels of 16 as an explicit panel width that the Gram never takes)."""
    import torch
    m = 40009
    At = workloads.gaussian(m, n, seed=850 + n)
    if kind == "repeated":
        At[n - 1] = At[1]
    elif kind == "zero":
        At[33] = 0.0
    elif kind == "nan":
        At[35, 12345] = float("nan")
    else:
        At = workloads.conditioned(m, n, 1e8, seed=n)  # served: no hand-over
    Ad = At.cuda().T
    T.tsqr_get_device_status()
    R = T.tsqr_r(Ad)
    status = T.tsqr_get_device_status()
    assert status == (T.STATUS_NONFINITE if kind == "nan" else T.SUCCESS)
    if kind == "kappa":
        _check(oracle, R, At)
    elif n < 56:
        ref = T.tsqr_r_ex(Ad, plan=T.make_plan("hybrid"))
        assert torch.equal(torch.nan_to_num(R), torch.nan_to_num(ref))
    if kind in ("repeated", "zero"):
        assert np.all(np.diag(R.cpu().numpy()) >= 0)
        assert oracle.gram_residual(oracle.from_torch_colmajor(At), R.cpu().numpy(), nthreads=16) <= 1e-13


@pytest.mark.parametrize("m,n,k,pad", [(2048, 31, 1, 0), (30011, 32, 1, 1), (20000, 8, 2, 0),
                                       (50001, 96, 24, 3), (40000, 55, 1, 0)])
def test_least_squares_of_two_matrices(oracle, T, m, n, k, pad):
    """[A | B] summed where A and B are; X against the oracle's least squares."""
    import torch
    At = workloads.gaussian(m, n, seed=n)
    Bt = workloads.gaussian(m, k, seed=k + 1)
    big = torch.full((n, m + pad), float("nan"), dtype=torch.float64)
    big[:, :m] = At
    X, R = T.tsqr_lstsq(big.cuda().T[:m, :], Bt.cuda().T)
    _check(oracle, R, At)
    A, B = oracle.from_torch_colmajor(At), oracle.from_torch_colmajor(Bt)
    Xo = oracle.lstsq(A, B, nthreads=16)
    kap = oracle.kappa_from_r(oracle.householder_r(A, nthreads=16))
    res = np.linalg.norm(B - A @ Xo)
    tol = max(50.0, 2.0 * np.sqrt(m)) * (kap + kap ** 2 * res /
                                         (np.linalg.norm(A, 2) * np.linalg.norm(Xo))) * U
    assert np.linalg.norm(X.cpu().numpy() - Xo) <= tol * np.linalg.norm(Xo)
    At[n // 2] = At[0]  # dependent: the copy and the Householder reduction behind the sum
    T.tsqr_get_device_status()
    X, R = T.tsqr_lstsq(At.cuda().T, Bt.cuda().T)
    T.tsqr_get_device_status()
    assert oracle.gram_residual(oracle.from_torch_colmajor(At), R.cpu().numpy(), nthreads=16) <= 1e-13


def test_batch_served_and_handed_over(oracle, T):
    """A batch of matrices the sum serves (one and several column blocks, ragged), matrices it is
    not tried on (too few rows), and matrices it hands over (a zero column, a repeated one, NaN)."""
    import torch
    g = torch.Generator().manual_seed(31)
    ms = [300, 4097, 70001, 20000, 513, 255, 100, 0, 9000, 8192, 5000, 40000, 260, 3000]
    ns = [5, 16, 33, 64, 128, 8, 64, 4, 24, 40, 7, 100, 65, 1]
    bad = {8: "zero", 9: "repeated", 10: "nan"}
    offs = [0]
    for m, n in zip(ms, ns):
        offs.append(offs[-1] + m * n)
    buf = torch.randn(offs[-1], generator=g, dtype=torch.float64)
    for i, kind in bad.items():
        A = buf[offs[i]:offs[i + 1]].view(ns[i], ms[i])
        if kind == "zero":
            A[3] = 0.0
        elif kind == "repeated":
            A[ns[i] - 1] = A[0]
        else:
            A[2, 77] = float("nan")
    bd = buf.cuda()
    roff = [0]
    for n in ns:
        roff.append(roff[-1] + n * n)
    ptrs = [bd.data_ptr() + 8 * o for o in offs[:-1]]
    T.tsqr_get_device_status()
    R = torch.full((roff[-1],), float("nan"), dtype=torch.float64, device="cuda")
    T.tsqr_r_batched(ptrs, ms, ns, roff, R)
    assert T.last_batch_plan().leaf == T.LEAF_GRAM
    assert T.tsqr_get_device_status() == T.STATUS_NONFINITE
    again = torch.zeros_like(R)
    T.tsqr_r_batched(ptrs, ms, ns, roff, again, plan=T.last_batch_plan())
    assert torch.equal(torch.nan_to_num(again), torch.nan_to_num(R))
    T.tsqr_get_device_status()  # clears it
    for i, (m, n) in enumerate(zip(ms, ns)):
        Ri = R[roff[i]:roff[i + 1]].view(n, n).T
        At = buf[offs[i]:offs[i + 1]].view(n, m)
        if bad.get(i) == "nan":
            assert not torch.isfinite(Ri).all()
        elif m == 0:
            assert torch.all(Ri == 0)
        elif i in bad or m < 4 * n:
            assert oracle.gram_residual(oracle.from_torch_colmajor(At), Ri.cpu().numpy()) <= 1e-13
        else:
            _check(oracle, Ri, At)


@pytest.mark.parametrize("m,n", [(520, 129), (1100, 160), (20000, 200), (9001, 290), (5000, 512)])
def test_wide_factor(oracle, T, m, n):
    """Past 128 columns the summed Gram is factored by block rows; bounds of the panels' tests."""
    At = workloads.gaussian(m, n, seed=n)
    A = oracle.from_torch_colmajor(At)
    R = T.tsqr_caqr_r(At.cuda().T).cpu().numpy()
    Ro = oracle.householder_r(A, nthreads=16)
    assert np.all(np.tril(R, -1) == 0) and np.all(np.diag(R) >= 0)
    c = max(50.0, 2.0 * np.sqrt(m * n / 32.0))
    np.testing.assert_allclose(R, Ro, rtol=0, atol=c * oracle.kappa_from_r(Ro) * U * np.linalg.norm(Ro))
    assert oracle.gram_residual(A, R, nthreads=16) <= 1e-13


@pytest.mark.parametrize("kind", ["repeated", "nan", "kappa"])
def test_wide_handed_over(oracle, T, kind):
    m, n = 12001, 180
    At = workloads.gaussian(m, n, seed=77)
    if kind == "repeated":
        At[170] = At[3]
    elif kind == "nan":
        At[100, 5000] = float("nan")
    else:
        At = workloads.conditioned(m, n, 1e8, seed=7)
    T.tsqr_get_device_status()
    R = T.tsqr_caqr_r(At.cuda().T).cpu().numpy()
    assert T.tsqr_get_device_status() == (T.STATUS_NONFINITE if kind == "nan" else T.SUCCESS)
    if kind != "nan":
        assert oracle.gram_residual(oracle.from_torch_colmajor(At), R, nthreads=16) <= 1e-13


def test_batches_in_flight_keep_their_tables(T):
    """Two batches in turn on one stream with nothing waited for: each call's table of problems (some
    100 KB here) has to last until the device has read it, also after the call has returned."""
    import torch
    calls = []
    for seed in (1, 2):
        buf, ms, ns, offs = workloads.varlen_batch(700, 300, 3000, seed=seed, device="cuda")
        roff = [0]
        for n in ns:
            roff.append(roff[-1] + n * n)
        ptrs = [buf.data_ptr() + 8 * o for o in offs[:-1]]
        ref = torch.zeros(roff[-1], dtype=torch.float64, device="cuda")
        T.tsqr_r_batched(ptrs, ms, ns, roff, ref)
        torch.cuda.synchronize()
        calls.append((buf, ptrs, ms, ns, roff, ref))
    outs = []
    for k in range(12):
        buf, ptrs, ms, ns, roff, ref = calls[k % 2]
        outs.append(torch.zeros_like(ref))
        T.tsqr_r_batched(ptrs, ms, ns, roff, outs[-1])
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        assert torch.equal(out, calls[k % 2][5])


@pytest.mark.parametrize("m,n", [(256, 1), (512, 8), (513, 7), (1025, 8), (256, 9), (257, 16),
                                 (20479, 15), (257, 17), (12800, 24), (39041, 25), (19457, 32)])
def test_qr_from_the_gram_factor(oracle, T, m, n):
    """Q = A R^-1 at the edges of its tiles (512, 256 and 128 rows a tile for up to 8, 16 and 32
    columns, 152 tiles a wave) and width classes, leading dimensions padded; R is tsqr_r_ex's under
    the plan reported, and what the oracle gives."""
    import torch
    At = workloads.gaussian(m, n, seed=700 + n)
    big = torch.full((n, m + 3), float("nan"), dtype=torch.float64)
    big[:, :m] = At
    Ad = big.cuda().T[:m, :]
    Qbig = torch.full((n, m + 5), float("nan"), dtype=torch.float64, device="cuda")
    Q, R = T.tsqr_qr(Ad, Q=Qbig.T[:m, :])
    p = T.last_plan()
    assert p.leaf == T.LEAF_GRAM_Q
    assert torch.equal(T.tsqr_r_ex(Ad, plan=p), R)
    _check(oracle, R, At)
    Qo, Ro = oracle.householder_qr(oracle.from_torch_colmajor(At), nthreads=16)
    tol = max(50.0, 2.0 * np.sqrt(m)) * oracle.kappa_from_r(Ro) * U * np.linalg.norm(Qo)
    np.testing.assert_allclose(Q.cpu().numpy(), Qo, rtol=0, atol=tol)
    Qd = Q.cpu().numpy()
    assert np.abs(Qd.T @ Qd - np.eye(n)).max() <= 50 * U
    assert torch.isnan(Qbig[:, m:]).all()
    assert T.tsqr_get_device_status() == T.SUCCESS


@pytest.mark.parametrize("kind", ["kappa10", "kappa100", "kappa1e4", "outlier", "zeros", "integers"])
@pytest.mark.parametrize("n", [8, 13, 32])
def test_qr_value_ranges(oracle, T, n, kind):
    """On both sides of the line to the reflectors: conditions 10, 100 and 1e4, an entry 2^30 above
    the rest (a column its peak dominates), rows of zeros, small whole numbers.  Orthonormal to
    50 u and A = Q R to c(m) u either way."""
    import torch
    m = 50001
    if kind.startswith("kappa"):
        At = workloads.conditioned(m, n, float(kind[5:]), seed=n)
    else:
        At = workloads.gaussian(m, n, seed=720 + n)
    if kind == "outlier":
        At[:, m // 2] *= 2.0 ** 30
        At[1, m // 2] = 1.0
    elif kind == "zeros":
        At[:, 1000:40000] = 0.0
    elif kind == "integers":
        At = torch.round(At * 4.0)
    Ad = At.cuda().T
    Q, R = T.tsqr_qr(Ad)
    assert torch.equal(T.tsqr_r_ex(Ad, plan=T.last_plan()), R)
    A, Qh, Rh = oracle.from_torch_colmajor(At), Q.cpu().numpy(), R.cpu().numpy()
    assert np.abs(Qh.T @ Qh - np.eye(n)).max() <= 50 * U
    assert np.linalg.norm(A - Qh @ Rh) <= 2.0 * np.sqrt(m) * U * np.linalg.norm(A)
    if kind == "zeros":
        assert np.all(Qh[1000:40000] == 0)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_batch_repeated_after_another_call(T, dtype):
    """The same batch (same buffers) before and after a call that takes the same workspace, and
    after the replay of a graph that does: its problem table is its own each time."""
    import torch
    dt = torch.float64 if dtype == "f64" else torch.float32
    ms, ns = [600 + 37 * i for i in range(24)], [(8, 16, 32, 64)[i % 4] for i in range(24)]
    offs, roff = [0], [0]
    for m, n in zip(ms, ns):
        offs.append(offs[-1] + m * n)
        roff.append(roff[-1] + n * n)
    g = torch.Generator(device="cuda").manual_seed(5)
    buf = torch.randn(offs[-1], generator=g, dtype=dt, device="cuda")
    wide = torch.randn(128, 60000, generator=g, dtype=torch.float64, device="cuda").T
    code = (T.F64, T.PREC_F64) if dtype == "f64" else (T.F32, T.PREC_MIXED)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())

    def batch():
        R = torch.empty(roff[-1], dtype=torch.float64, device="cuda")
        T.tsqr_r_batched([buf.data_ptr() + buf.element_size() * o for o in offs[:-1]], ms, ns, roff,
                         R, dtype=code[0], prec=code[1])
        return R

    with torch.cuda.stream(s):
        Rw = T.tsqr_r(wide)  # the workspace at its full size before the first table
        first = batch()
        T.tsqr_r(wide, R=Rw)
        second = batch()
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            T.tsqr_r(wide, R=Rw)
        third = batch()
        graph.replay()
        fourth = batch()
    s.synchronize()
    for R in (second, third, fourth):
        assert torch.equal(first, R)


@pytest.mark.parametrize("n", [7, 32, 40, 64])
def test_hand_over_under_capture(T, n):
    """A captured call whose replays are served and handed over in turn (the Householder reduction
    takes the shared memory that the sum's barriers stood in): each replay gives the direct call's
    bytes."""
    import torch
    m = 30011
    good = workloads.gaussian(m, n, seed=860 + n).cuda()
    zero, repeated = good.clone(), good.clone()
    zero[n // 2] = 0.0
    repeated[n - 1] = repeated[0]
    ref = [T.tsqr_r(A.T).clone() for A in (good, zero, repeated)]
    buf, out = good.clone(), T.empty_r(n, "cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        T.tsqr_r(buf.T, R=out)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        T.tsqr_r(buf.T, R=out, stream=s)
    for k in (0, 1, 0, 2, 1, 2, 0):
        buf.copy_((good, zero, repeated)[k])
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref[k]), k
    assert T.tsqr_get_device_status() == T.SUCCESS


def test_wide_handed_over_on_streams(oracle, T):
    """A dependent column in the first block row of the wide factor, found by every CTA of that
    launch, with other calls of the kind on two more streams (CTAs start late): the same bytes each
    time, and A's Gram."""
    import torch
    m, n = 3000, 700
    At = workloads.gaussian(m, n, seed=78)
    At[9] = At[4]
    Ad = At.cuda().T
    ref = T.tsqr_caqr_r(Ad).clone()
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = []
    for st in streams * 3:
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            outs.append(T.tsqr_caqr_r(Ad))
    torch.cuda.synchronize()
    for R in outs:
        assert torch.equal(R, ref)
    assert oracle.gram_residual(oracle.from_torch_colmajor(At), ref.cpu().numpy(), nthreads=16) <= 1e-13


@pytest.mark.parametrize("p", [-396, -405, -430, -460])
@pytest.mark.parametrize("which", ["one", "all"])
@pytest.mark.parametrize("call,m,n", [("r", 4096, 4), ("r", 20011, 32), ("r", 20011, 40),
                                      ("r", 20011, 100), ("host", 9001, 12), ("qr", 20011, 16),
                                      ("caqr", 6007, 180), ("lstsq", 20011, 20), ("batch", 4096, 33)])
def test_columns_of_small_scale(oracle, T, call, m, n, which, p):
    """Columns whose largest entry is at 2^p, about the least the fixed point serves (2^-400) and
    below: column j of R scales with column j of A exactly, so R scaled back meets the unscaled
    matrix's bounds, whichever reduction gave it."""
    import torch
    At = workloads.gaussian(m, n, seed=900 + n)
    e = torch.zeros(n, dtype=torch.float64)
    if which == "one":
        e[n // 2] = p
    else:
        e[:] = p
    S = torch.exp2(e)
    As = (At * S[:, None]).contiguous()
    T.tsqr_get_device_status()
    if call == "r":
        R = T.tsqr_r(As.cuda().T)
    elif call == "host":
        R = T.tsqr_r_host(As.pin_memory().T)
        torch.cuda.synchronize()
    elif call == "caqr":
        R = T.tsqr_caqr_r(As.cuda().T)
    elif call == "qr":
        Q, R = T.tsqr_qr(As.cuda().T)
        Qh = Q.cpu().numpy()
        assert np.abs(Qh.T @ Qh - np.eye(n)).max() <= 50 * U
    elif call == "lstsq":
        Bt = workloads.gaussian(m, 2, seed=5)  # the second right-hand side of the columns' scale
        X, R = T.tsqr_lstsq(As.cuda().T, (Bt * torch.exp2(
            torch.tensor([0.0, p], dtype=torch.float64))[:, None]).cuda().T)
        A, B = oracle.from_torch_colmajor(At), oracle.from_torch_colmajor(Bt)
        Xo = oracle.lstsq(A, B, nthreads=16)
        Xh = X.cpu().numpy() * S.numpy()[:, None] * np.exp2([0.0, -p])
        kap = oracle.kappa_from_r(oracle.householder_r(A, nthreads=16))
        tol = 2.0 * np.sqrt(m) * (kap + kap ** 2 * np.linalg.norm(B - A @ Xo) /
                                  (np.linalg.norm(A, 2) * np.linalg.norm(Xo))) * U
        assert np.linalg.norm(Xh - Xo) <= tol * np.linalg.norm(Xo)
    else:
        buf = torch.cat([workloads.gaussian(m, n, seed=1).reshape(-1), As.reshape(-1)]).cuda()
        out = torch.empty(2 * n * n, dtype=torch.float64, device="cuda")
        T.tsqr_r_batched([buf.data_ptr(), buf.data_ptr() + 8 * m * n], [m, m], [n, n],
                         [0, n * n, 2 * n * n], out)
        R = out[n * n:].view(n, n).T
    assert T.tsqr_get_device_status() == T.SUCCESS
    _check(oracle, R.cpu() * torch.exp2(-e)[None, :], At)


@pytest.mark.parametrize("call", ["r", "qr", "lstsq", "batch"])
def test_rows_past_what_128_bits_hold(T, call):
    """402,653,184 rows of 1.75, every slab's first block (which sets the exponent) four times
    smaller: the squares' sum is 1.15 2^128 in the units of a slab.  Two columns, the second with
    signs in turn: orthogonal, so R is the norm times I, within c(m) u."""
    import torch
    m = 3 << 27
    slabs = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    At = torch.full((2, m), 1.75, dtype=torch.float64, device="cuda")
    first = torch.arange(slabs, device="cuda") * (m // 64) // slabs
    At.view(2, m // 64, 64)[:, first] = 0.4375
    At[1, 1::2] *= -1.0
    norm = np.sqrt((m - 64 * slabs) * 1.75 ** 2 + 64 * slabs * 0.4375 ** 2)
    tol = 2.0 * np.sqrt(m) * U
    T.tsqr_get_device_status()
    if call == "r":
        R = T.tsqr_r(At.T)
    elif call == "qr":
        Q, R = T.tsqr_qr(At.T)
        At *= 1.0 / norm
        assert (Q.T - At).abs().max().item() <= tol / np.sqrt(m)
    elif call == "lstsq":
        B = At[1:].clone()
        B[:, :m // 8] = At[0, :m // 8]  # an eighth of the first column's square, the rest orthogonal
        X, R = T.tsqr_lstsq(At[:1].T, B.T)
        assert abs(X.item() - 0.125) <= 4.0 * tol and abs(R.item() - norm) <= tol * norm
        return
    else:
        R = torch.empty(4, dtype=torch.float64, device="cuda")
        T.tsqr_r_batched([At.data_ptr()], [m], [2], [0, 4], R)
        R = R.view(2, 2).T
    assert T.tsqr_get_device_status() == T.SUCCESS
    assert (R.cpu() - norm * torch.eye(2, dtype=torch.float64)).abs().max().item() <= tol * norm


@pytest.mark.parametrize("n", [8, 16, 24, 32, 40])
def test_same_bytes_where_exponents_rise(T, n):
    """One column whose peaks (2^6, 2^10, ...: its exponent rises twelve times in a slab, at other
    places in each) break the rounds off, beside columns of condition 1e9, whose last pivots magnify
    a difference in how their sums are cut: the same bytes on every run, alone and beside other
    work."""
    import torch
    blocks = 300 if n > 8 else 700
    m = 152 * 64 * blocks
    g = torch.Generator(device="cuda").manual_seed(n)
    V = torch.linalg.qr(torch.randn(n - 1, n - 1, dtype=torch.float64, device="cuda", generator=g))[0]
    s = torch.logspace(0, -9, n - 1, dtype=torch.float64, device="cuda")
    At = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g)
    At[:-1] = (V * s) @ At[:-1]
    gc = torch.Generator().manual_seed(n)
    for slab in range(152):
        peaks = torch.randperm(blocks - 20, generator=gc)[:12].sort().values + 10
        At[-1, ((slab * blocks + peaks) * 64 + 11).cuda()] = torch.exp2(
            6 + 4 * torch.arange(12, dtype=torch.float64)).cuda()
    ref = T.tsqr_r(At.T).clone()
    side, noise = torch.cuda.Stream(), torch.randn(2048, 2048, device="cuda")
    outs = []
    for k in range(60):
        if k % 3 == 0:
            with torch.cuda.stream(side):
                noise = noise @ noise * 1e-3
        outs.append(T.tsqr_r(At.T))
    torch.cuda.synchronize()
    assert sum(not torch.equal(R, ref) for R in outs) == 0
    assert T.tsqr_get_device_status() == T.SUCCESS


@pytest.mark.parametrize("m,n,k", [(20011, 20, 1), (9001, 40, 2), (9001, 60, 3), (20011, 96, 24)])
@pytest.mark.parametrize("kind", ["served", "handed over"])
def test_least_squares_plans_go_back(T, m, n, k, kind):
    """The plan least squares reports gives the same bytes when it is passed back (on both sides of 56
    columns of [A | B]), served or handed over; so does tsqr_r's, where that is the sum's."""
    import torch
    At = workloads.gaussian(m, n, seed=n)
    if kind == "handed over":
        At[n - 1] = At[0]
    A, B = At.cuda().T, workloads.gaussian(m, k, seed=k).cuda().T
    T.tsqr_r(A)
    pr = T.last_plan()
    X, R = T.tsqr_lstsq(A, B)
    p = T.last_plan()
    assert (p.tree, p.leaf) == (T.TREE_HYBRID, T.LEAF_GRAM) and p.tile_rows > 0
    for plan in [p] + ([pr] if pr.leaf == T.LEAF_GRAM else []):
        X1, R1 = T.tsqr_lstsq(A, B, plan=plan)
        assert torch.equal(R1, R) and torch.equal(torch.nan_to_num(X1), torch.nan_to_num(X))
    bad = T.make_plan("binary", tile_rows=256)
    bad.leaf = T.LEAF_GRAM
    for A1, B1, plan in [(A, B, bad), (A[:200], B[:200], p)]:  # no tree of the sum's, too few rows
        with pytest.raises(T.TsqrError) as e:
            T.tsqr_lstsq(A1, B1, plan=plan)
        assert e.value.status == T.ERR_INVALID_ARG
    T.tsqr_get_device_status()  # clears it


@pytest.mark.parametrize("m,n,panel", [(9001, 12, 0), (9001, 12, 16), (20011, 40, 64)])
@pytest.mark.parametrize("kind", ["served", "handed over"])
def test_one_panel_plans_go_back(T, m, n, panel, kind):
    """The plan tsqr_caqr_r reports for one panel gives the same bytes when it is passed back."""
    import torch
    At = workloads.gaussian(m, n, seed=n)
    if kind == "handed over":
        At[n - 1] = At[0]
    A = At.cuda().T
    R = T.tsqr_caqr_r(A, panel=panel)
    p = T.last_plan()
    assert p.leaf == T.LEAF_GRAM
    assert torch.equal(T.tsqr_caqr_r(A, panel=panel, plan=p), R)


@pytest.mark.parametrize("m,n", [(40009, 56), (40000, 64), (30011, 80), (100003, 96), (65537, 128),
                                 (12001, 180)])
def test_householder_panels_on_request(oracle, T, m, n):
    """Panels of the default width without the sum before them (leaf FOLD): within parity of the
    oracle on a matrix the sum serves; and the bytes of AUTO's call on matrices it hands over."""
    import torch
    plan = T.make_plan("panels", tile_rows=16, leaf="fold")
    At = workloads.gaussian(m, n, seed=n + 1)
    R = T.tsqr_r_ex(At.cuda().T, plan=plan)
    p = T.last_plan()
    assert (p.tree, p.tile_rows, p.leaf) == (T.TREE_PANELS, 16, T.LEAF_FOLD)
    if n <= 128:
        r = T.tsqr_resolve_plan(m, n, plan=plan)
        assert (r.tree, r.tile_rows, r.leaf) == (T.TREE_PANELS, 16, T.LEAF_FOLD)
        _check(oracle, R, At)
    served = T.tsqr_r(At.cuda().T)
    assert T.last_plan().leaf == 0 and not torch.equal(R, served)
    for kind in ("repeated", "zero", "nan"):
        B = At.clone()
        if kind == "repeated":
            B[n - 2] = B[1]
        elif kind == "zero":
            B[n // 2] = 0.0
        else:
            B[n - 3, m // 2] = float("nan")
        T.tsqr_get_device_status()
        Ra = T.tsqr_r(B.cuda().T)
        sa = T.tsqr_get_device_status()
        Rb = T.tsqr_r_ex(B.cuda().T, plan=plan)
        assert sa == T.tsqr_get_device_status()
        assert torch.equal(torch.nan_to_num(Ra), torch.nan_to_num(Rb)), kind
        assert torch.equal(torch.isfinite(Ra), torch.isfinite(Rb)), kind


def _batch_call(T, count=24, m0=600):
    """A small FP64 batch: (call(stream) -> R, R's reference)."""
    import torch
    ms, ns = [m0 + 37 * i for i in range(count)], [(8, 16, 32, 40)[i % 4] for i in range(count)]
    offs, roff = [0], [0]
    for m, n in zip(ms, ns):
        offs.append(offs[-1] + m * n)
        roff.append(roff[-1] + n * n)
    g = torch.Generator(device="cuda").manual_seed(count)
    buf = torch.randn(offs[-1], generator=g, dtype=torch.float64, device="cuda")
    ptrs = [buf.data_ptr() + 8 * o for o in offs[:-1]]

    def call(R, stream):
        T.tsqr_r_batched(ptrs, ms, ns, roff, R, stream=stream)

    ref = torch.empty(roff[-1], dtype=torch.float64, device="cuda")
    call(ref, None)
    torch.cuda.synchronize()
    return call, ref, buf


def test_batch_beside_a_capture_of_another_thread(T):
    """One thread captures a graph in the strictest mode while another runs batches on a stream of its
    own (whose workspace is there; their tables are new): both succeed."""
    import threading

    import torch
    call, ref, _keep = _batch_call(T)
    x = torch.ones(1000, device="cuda")
    outs = [torch.zeros_like(ref) for _ in range(8)]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    errors = []
    call(outs[0], s2)

    def work():
        try:
            for R in outs:
                call(R, s2)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s1, capture_error_mode="global"):
        x += 1.0
        t = threading.Thread(target=work)
        t.start()
        t.join()
        x += 1.0
    g.replay()
    torch.cuda.synchronize()
    assert not errors
    assert (x == 3.0).all()
    for R in outs:
        assert torch.equal(R, ref)


def test_batch_calls_do_not_wait_for_the_stream(T):
    """Thirty batch calls, small and larger tables in turn, on a stream that is busy for some 0.2 s:
    the calls return while it is; and a second thirty with the slots at hand."""
    import time

    import torch
    small, large = _batch_call(T), _batch_call(T, count=900, m0=260)
    outs = [torch.zeros_like(b[1]) for b in (small, large)]
    s = torch.cuda.Stream()
    for (call, _, _), out in zip((small, large), outs):  # the workspace at its full size
        call(out, s)
    for _ in range(2):
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            torch.cuda._sleep(400_000_000)
        t0 = time.perf_counter()
        for k in range(30):
            (small, large)[k % 2][0](outs[k % 2], s)
        took = time.perf_counter() - t0
        assert not s.query() and took < 0.15, took
    torch.cuda.synchronize()
    for (_, ref, _), out in zip((small, large), outs):
        assert torch.equal(out, ref)


def test_captured_batches_give_their_tables_back(T):
    """Sixty graphs of a batch with a table of 1.3 MB, each replayed, and left while its last replay
    is on its way: the process does not grow by their tables (78 MB)."""
    import gc
    import os

    import torch
    n, m, count = 8, 260, 6000
    buf = torch.randn(count * m * n, dtype=torch.float64, device="cuda")
    args = ([buf.data_ptr() + 8 * m * n * i for i in range(count)], [m] * count, [n] * count,
            [n * n * i for i in range(count + 1)])
    R = torch.empty(count * n * n, dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    T.tsqr_r_batched(*args, R, stream=s)
    torch.cuda.synchronize()
    ref = R.clone()

    def resident():
        gc.collect()
        with open("/proc/self/statm") as f:
            return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")

    before = 0
    for k in range(65):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            T.tsqr_r_batched(*args, R, stream=s)
        R.zero_()
        g.replay()
        g.replay()
        del g
        torch.cuda.synchronize()
        assert torch.equal(R, ref)
        if k == 4:
            before = resident()
    assert resident() - before < 20 << 20


@pytest.mark.parametrize("n", range(1, 33))
def test_chunks_behind_the_sum(T, n):
    """The Householder leaves behind the single launch fold chunks that fill shared memory where there
    are rows for it (four tenths of an SM's, a number of rows that blocks well), and where there are
    not, as many leaves as chunks of the least height (two rows a lane) give."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = T.tsqr_resolve_plan(1 << 24, n)
    assert p.leaf == T.LEAF_GRAM
    per_sm = -(-p.ctas // sms)
    assert p.ctas == per_sm * sms and per_sm * p.tile_rows * n * 8 >= 0.4 * 227 * 1024
    for m in (10000, 100003):
        p = T.tsqr_resolve_plan(m, n)
        assert p.ctas >= min(0.8 * sms, m // (64 * p.warps))


@pytest.mark.parametrize("m", [256, 300, 641, 1000, 5003, 60013, 400009])
@pytest.mark.parametrize("n", [1, 2, 5, 8, 9, 16, 24, 32])
def test_leaves_behind_the_sum(T, m, n):
    """The Householder leaves of the single launch, three a CTA, at every block height (one, two and
    three rows) and with fewer leaves than groups: the bytes of that reduction by itself."""
    import torch
    At = workloads.gaussian(m, n, seed=m % 89 + n)
    At[n // 2] = 0.0
    Ad = At.cuda().T
    R = T.tsqr_r(Ad)
    p = T.last_plan()
    assert p.leaf == T.LEAF_GRAM and p.warps == 4 and T.tsqr_last_launch_count() == 1
    ref = T.tsqr_r_ex(Ad, plan=T.make_plan("hybrid", tile_rows=p.tile_rows, ctas=p.ctas,
                                           warps=p.warps, arity=p.arity))
    assert torch.equal(R, ref)
    assert T.tsqr_get_device_status() == T.SUCCESS


@pytest.mark.parametrize("m,n,k", [(9001, 8, 2), (20011, 31, 1), (20011, 32, 1), (20011, 33, 8),
                                   (9001, 60, 5), (20011, 100, 25), (6007, 150, 40), (5003, 128, 33)])
@pytest.mark.parametrize("kind", ["consistent", "one of them", "noisy", "tiny"])
def test_regressions_need_only_the_pivots_of_the_matrix(oracle, T, m, n, k, kind):
    """B in the range of A (whose residual has no pivot in the sum): served, X as close to the known
    solution as for a noisy B, R the same bytes whatever B is.  B below the fixed point's range
    goes to the Householder reduction."""
    import torch
    At = workloads.gaussian(m, n, seed=n)
    X0 = torch.randn(n, k, generator=torch.Generator().manual_seed(3), dtype=torch.float64)
    Bt = (At.T @ X0).T.contiguous()
    if kind == "noisy":
        Bt += workloads.gaussian(m, k, seed=5)
    elif kind == "one of them":
        Bt[1:] += workloads.gaussian(m, k, seed=5)[1:]
    elif kind == "tiny":
        Bt[0] *= 2.0 ** -430
        X0[:, 0] *= 2.0 ** -430
    T.tsqr_get_device_status()
    X, R = T.tsqr_lstsq(At.cuda().T, Bt.cuda().T)
    assert T.tsqr_get_device_status() == T.SUCCESS
    A, B = oracle.from_torch_colmajor(At), oracle.from_torch_colmajor(Bt)
    X, X0 = X.cpu().numpy(), X0.numpy()
    kap = oracle.kappa_from_r(oracle.householder_r(A, nthreads=16))
    c = max(50.0, 2.0 * np.sqrt(m * max(1.0, n / 32.0)))
    for j in range(k):
        ref = X0[:, j]
        if kind == "noisy" or (kind == "one of them" and j > 0):
            ref = oracle.lstsq(A, np.asfortranarray(B[:, j:j + 1]), nthreads=16)[:, 0]
        res = np.linalg.norm(B[:, j] - A @ ref)
        tol = c * (kap + kap ** 2 * res / (np.linalg.norm(A, 2) * np.linalg.norm(ref))) * U
        assert np.linalg.norm(X[:, j] - ref) <= tol * np.linalg.norm(ref)
    if kind != "tiny":
        noisy = workloads.gaussian(m, k, seed=6)
        assert torch.equal(T.tsqr_lstsq(At.cuda().T, noisy.cuda().T)[1], R)
    if n + k <= 128:
        _check(oracle, R, At)
