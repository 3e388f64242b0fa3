"""The fp64 contraction kernel and the factorisations / solves of both precisions at the edges of their tiles (fp64: 64 x 64
and 32 x 64 tiles, K slabs of 16, block columns of 64; fp32: block columns of 128), against plain fp64 torch."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _api():
    from paper_2510_03246_b200 import api
    return api


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("transA", [False, True])
@pytest.mark.parametrize("transB", [False, True])
@pytest.mark.parametrize("M,N,K,pad", [(1, 1, 1, 0), (33, 65, 17, 1), (64, 64, 16, 0), (130, 70, 250, 3), (1027, 769, 131, 2),
                                       (2048, 832, 64, 4)])
def test_gemm_fp64_accumulation(dtype, transA, transB, M, N, K, pad):
    """Every stored orientation, aligned and unaligned pitches, accumulation into C and the lower triangle alone."""
    api = _api()
    g = torch.Generator(device="cuda").manual_seed(M + 7 * N + 13 * K)

    def stored(r, c):
        buf = torch.randn(r, c + pad, generator=g, device="cuda", dtype=torch.float64).to(dtype)
        return buf[:, :c]

    A, B = stored(*((K, M) if transA else (M, K))), stored(*((N, K) if transB else (K, N)))
    C0 = stored(M, N)
    a, b = (A.T if transA else A).double(), (B.T if transB else B).double()
    want = 0.75 * (a @ b) - 0.5 * C0.double()
    # one rounding to the stored type, and K + 2 roundings of the fp64 sum on either side
    unit = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -53
    bound = unit * want.abs() + 2 * (K + 4) * 2.0 ** -53 * (a.abs() @ b.abs() + C0.double().abs())
    got = C0.clone()
    api.sp_gemm(A, B, got, transA, transB, alpha=0.75, beta=-0.5)
    assert bool(((got.double() - want).abs() <= bound).all())
    low = C0.clone()
    api.sp_gemm(A, B, low, transA, transB, alpha=0.75, beta=-0.5, lower_only=True)
    tri = torch.ones(M, N, device="cuda", dtype=torch.bool).tril()
    assert torch.equal(low[tri], got[tri])


@pytest.mark.parametrize("a_kmajor", [False, True])
@pytest.mark.parametrize("b_kmajor", [False, True])
@pytest.mark.parametrize("M,N,K,lower", [(8, 8, 8, False), (256, 128, 64, False), (264, 136, 72, False), (1000, 64, 704, False),
                                         (1288, 256, 768, True), (520, 520, 128, False), (2304, 1032, 320, False),
                                         (3000, 256, 192, False)])
def test_gemm_tensor_core_tiles_of_both_widths(a_kmajor, b_kmajor, M, N, K, lower):
    """256 x 128 tiles (few tiles, or few columns) and 256 x 256 tiles, stored and accumulated into C."""
    api = _api()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(*((M, K) if a_kmajor else (K, M)), generator=g, device="cuda").bfloat16()
    B = torch.randn(*((N, K) if b_kmajor else (K, N)), generator=g, device="cuda").bfloat16()
    a, b = (A if a_kmajor else A.T).double(), (B.T if b_kmajor else B).double()
    C0 = torch.randn(M, N, generator=g, device="cuda")
    # exact products, fp32 sums: at most one rounding of 2^-23 (the unit truncates) of the sum of magnitudes per term
    bound = (K + 2) * 2.0 ** -23 * (a.abs() @ b.abs() + C0.double().abs())
    keep = torch.ones(M, N, dtype=torch.bool, device="cuda")
    if lower:
        keep = keep.tril()
    for beta, dtype in ((0.0, torch.float32), (1.0, torch.float32), (0.0, torch.bfloat16)):
        C = C0.to(dtype)
        want = a @ b + beta * C.double()
        api.sp_gemm(A, B, C, not a_kmajor, b_kmajor, beta=beta, lower_only=lower, use_tensor_cores=True)
        off = (C.double() - want).abs() - bound - (2.0 ** -8 * want.abs() if dtype == torch.bfloat16 else 0)
        assert float(off[keep].max()) <= 0


@pytest.mark.parametrize("M,N,K,lower", [(256, 256, 64, True), (128, 96, 64, True), (1288, 256, 768, True), (520, 520, 128, True),
                                         (256, 256, 64, False)])
def test_profile_counts_the_operations_of_a_lower_triangle(M, N, K, lower):
    """The triangle of the leading N x N square and the rows below it, whichever tile computes them."""
    api = _api()
    A, B = (torch.ones(r, K, device="cuda", dtype=torch.bfloat16) for r in (M, N))
    C = torch.zeros(M, N, device="cuda")
    api.sp_profile_begin(1)
    try:
        api.sp_gemm(A, B, C, False, True, lower_only=lower, use_tensor_cores=True)
        torch.cuda.synchronize()
        got = api.sp_profile_read()["gemm_tc"]
    finally:
        api.sp_profile_begin(0)
    assert got["records"] == 1 and got["flops"] == (K * N * (2 * M - N) if lower else 2 * M * N * K)


def _spd(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(2 * n + 3, n, generator=g, device="cuda") * torch.logspace(0, 1.5, n, device="cuda")
    G = (X.T @ X).float()
    return torch.tril(G) + torch.tril(G, -1).T


@pytest.mark.parametrize("n,m", [(1, 1), (3, 70), (63, 5), (64, 64), (65, 33), (127, 129), (200, 1), (321, 500), (1030, 259)])
def test_precise_ridge_solve_at_block_edges(n, m):
    api = _api()
    G = _spd(n, n)
    R = torch.randn(m, n, generator=torch.Generator(device="cuda").manual_seed(m), device="cuda")
    got = api.sp_ridge_solve(R, G, 0.01, True, precise=True)
    H = G.double() + 0.01 * G.double().diagonal().mean() * torch.eye(n, device="cuda", dtype=torch.float64)
    want = torch.linalg.solve(H, R.double().T).T
    # fp64 throughout (condition number below 1e5: 1e-10 of the largest entry), stored as fp32 (2^-24)
    assert float((got.double() - want).abs().max() / want.abs().max()) < 1.2e-7
    again = api.sp_ridge_solve(R, G, 0.01, True, precise=True)
    assert torch.equal(got, again)      # no result depends on the order of the two streams


@pytest.mark.parametrize("n,m,k", [(64, 200, 64), (65, 200, 64), (3073, 1, 3073), (3073, 2, 3073), (3400, 491, 3400), (3400, 492, 3400),
                                   (3600, 400, 3300), (4097, 1600, 4096)])
def test_precise_solves_by_sweep_and_by_inverse(n, m, k):
    """Both sides of the lines between a backward sweep and the inverse of the factor; a refit narrower than the system whose
    workspace it has (k units of n kept), right up to that workspace's end."""
    api = _api()
    G = _spd(n, n)
    g = torch.Generator(device="cuda").manual_seed(m)
    R = torch.randn(m, n, generator=g, device="cuda")
    keep = torch.sort(torch.randperm(n, generator=g, device="cuda")[:k]).values
    mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    mask[keep] = 1
    rho = 0.01 * float(G.double().diagonal().mean())
    need = api.workspace_bytes(api.SP_WS_LINEAR_REFIT, m, n, 0, 0, api.SP_F64)
    buf = torch.full((need + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    got = api.sp_linear_refit(R, G, mask, k, rho, precise=True, ws=buf[:need])
    H = G[keep][:, keep].double() + rho * torch.eye(k, device="cuda", dtype=torch.float64)
    want = torch.linalg.solve(H, R[:, keep].double().T).T
    # fp64 throughout (condition number below 1e5: 1e-10 of the largest entry), stored as fp32 (2^-24)
    assert float((got[:, keep].double() - want).abs().max() / want.abs().max()) < 1.2e-7
    assert torch.all(got[:, mask == 0] == 0) and torch.all(buf[need:] == 0x5a)


@pytest.mark.parametrize("n,m", [(1, 3), (31, 40), (33, 8), (96, 129), (127, 64), (128, 200), (129, 7), (385, 96), (1000, 300)])
def test_tensor_core_ridge_solve_at_block_edges(n, m):
    """Diagonal blocks of 128 eliminated in sub-blocks of 32, panels of a few rows."""
    api = _api()
    G = _spd(n, n + 1)
    R = torch.randn(m, n, generator=torch.Generator(device="cuda").manual_seed(m), device="cuda")
    status = api.new_status(G.device)
    got = api.sp_ridge_solve(R, G, 0.1, True, status=status)
    H = G.double() + 0.1 * G.double().diagonal().mean() * torch.eye(n, device="cuda", dtype=torch.float64)
    want = torch.linalg.solve(H, R.double().T).T
    # backward stable fp32 solve: a few roundings of 2^-24 times the condition number (the ridge bounds it by 10 n)
    assert float((got.double() - want).abs().max() / want.abs().max()) < 4 * 2.0 ** -24 * 10 * max(n, 10)
    assert int(status[0]) == 0
    bad = G.clone()
    i = n // 2
    bad[i, i] = -bad[i, i].abs() * 100
    api.sp_ridge_solve(R, bad, 1e-6, False, status=status)
    assert status[:2].tolist() == [6, i]      # SP_ERR_NOT_SPD and the pivot


@pytest.mark.parametrize("n", [1, 2, 17, 31, 32, 33, 64, 65, 96, 97, 127])
def test_partial_diagonal_block_equals_the_whole_one(n):
    """A system that fills part of a diagonal block is eliminated up to its last sub-block only: the same bits as beside an
    identity that fills the block."""
    api = _api()
    G, R = _spd(n, n), torch.randn(70, n, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    whole, Rw = torch.eye(128, device="cuda"), torch.zeros(70, 128, device="cuda")
    whole[:n, :n], Rw[:, :n] = G, R
    got, want = api.sp_ridge_solve(R, G, 0.5, False), api.sp_ridge_solve(Rw, whole, 0.5, False)
    assert torch.equal(got, want[:, :n])


def _diagonal(lo, hi, n=128):
    """Diagonal matrix with entries over 2^lo .. 2^hi, mantissas spread."""
    e = torch.linspace(lo, hi, n, dtype=torch.float64, device="cuda")
    return torch.diag((2.0 ** e).float())


def test_reciprocal_square_roots_of_the_pivots():
    """A diagonal system solved for its own matrix: every entry of the answer is g y y with y = 1 / sqrt(g)."""
    api = _api()
    eye = torch.eye(128, device="cuda")
    # fp32: y to 2.5 x 2^-24, two products of 2^-24 each; at the upper end y^2 is subnormal (one more 2^-24 in y)
    for lo, hi, units in ((-100, 100, 7.0), (-125.5, 127.5, 9.0)):
        G = _diagonal(lo, hi)
        W = api.sp_ridge_solve(G, G, 0.0, False)
        assert torch.equal(W != 0, eye != 0)
        assert float((W.diagonal().double() - 1).abs().max()) <= units * 2.0 ** -24
    # fp64: a few 2^-53, nothing of which is left in fp32; subnormal fp32 entries among them
    G = _diagonal(-148.5, 127.5)
    assert torch.equal(api.sp_ridge_solve(G, G, 0.0, False, precise=True), eye)


@pytest.mark.parametrize("n", [5, 64, 130])
def test_precise_solve_with_extreme_pivots(n):
    """Pivots that are subnormal in fp64, near the upper end, or infinite (an accumulator that overflowed): the solution is what
    the square root and the division by it give, a column with an infinite pivot is zero."""
    api = _api()
    zero = torch.zeros(n, n, device="cuda")
    for rho, value in ((1e-310, 0.0), (5e-324, 0.0), (1e300, 3e38), (1.7e308, 3e38)):
        status = api.new_status(zero.device)
        W = api.sp_ridge_solve(torch.full_like(zero, value), zero, rho, False, precise=True, status=status)
        assert torch.equal(W, zero) and int(status[0]) == 0, rho
    G = _spd(n, n)
    R = torch.randn(7, n, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    i = n // 2
    rest = [j for j in range(n) if j != i]
    bad = G.clone()
    bad[i, i] = float("inf")
    W = api.sp_ridge_solve(R, bad, 0.5, False, precise=True)
    assert torch.equal(W[:, i], torch.zeros_like(W[:, i]))
    H = G[rest][:, rest].double() + 0.5 * torch.eye(n - 1, device="cuda", dtype=torch.float64)
    want = torch.linalg.solve(H, R[:, rest].double().T).T
    assert float((W[:, rest].double() - want).abs().max() / want.abs().max()) < 1.2e-7


@pytest.mark.parametrize("n,m", [(12288, 40), (12300, 200), (12420, 4800)])
def test_two_level_sweep_of_a_large_system(n, m):
    """Outer blocks of 512 columns, the last of them ragged; few right-hand sides (a block column pulls the update of the
    one before it) and more than one wave of panels holds (it does not)."""
    api = _api()
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(n + 64, n, generator=g, device="cuda")
    G = X.T @ X
    G = torch.tril(G) + torch.tril(G, -1).T
    del X
    R = torch.randn(m, n, generator=g, device="cuda")
    status = api.new_status(G.device)
    got = api.sp_ridge_solve(R, G, 0.1, True, status=status)
    assert int(status[0]) == 0
    # residual of the solution in fp64, relative to its terms: a few roundings of 2^-24 per block column (n / 128)
    H = G.double()
    H.diagonal().add_(0.1 * H.diagonal().mean())
    res = got.double() @ H - R.double()
    assert float(res.abs().max()) < (n // 128) * 2.0 ** -24 * float((got.double().abs() @ H.abs()).max())


@pytest.mark.parametrize("n,rows", [(4, 5), (64, 64), (72, 33), (200, 130), (1096, 70)])
def test_ordered_accumulators_come_back_in_channel_order(n, rows):
    """A module whose token pass works with the kept channels first: G_A (both triangles, from the lower one), R1 and R2 in
    channel order hold the entries of the ordered buffers, at the edges of the 32 x 32 tiles and of the 1024-column strips, and
    R1 is the product over the tokens."""
    api = _api()
    g = torch.Generator(device="cuda").manual_seed(n)
    d, N, k = 64, 8 * rows, max(1, n // 3)
    mod = api.FfnModule(torch.randn(N, d, generator=g, device="cuda").bfloat16(),
                        torch.randn(n, d, generator=g, device="cuda") * 0.1,
                        torch.randn(d, n, generator=g, device="cuda") * 0.1, overlap_k=k)
    mod.sp_ffn_init()
    mod.mask.zero_()
    mod.mask[torch.randperm(n, generator=g, device="cuda")[:k]] = 1
    p = api.AdmmParams(k_keep=k, rho=0.1, reselect_mask=False, skip_scores=True)
    for _ in range(2):
        mod.sp_admm_step(p)
    mod.check_status()
    want = mod.Z.double().T @ mod.X.double()
    # (Z enters the product as bf16: one rounding of 2^-9 per term)
    assert float((mod.R1.double() - want).abs().max()) < 2.0 ** -9 * float((mod.Z.double().abs().T @ mod.X.double().abs()).max())
    inv = torch.argsort(mod.decay_tag[8:8 + n])
    ordered = torch.tril(mod.G_A_perm) + torch.tril(mod.G_A_perm, -1).T
    assert torch.equal(mod.G_A, ordered[inv][:, inv])
    assert torch.equal(mod.R1, mod.R1_perm[inv]) and torch.equal(mod.R2, mod.R2_perm[:, inv])


@pytest.mark.parametrize("d", [8, 64, 72, 136, 520, 1096])
def test_cached_input_inverse_at_block_edges(d):
    api = _api()
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(2 * d, d, generator=g, device="cuda").bfloat16()
    mod = api.FfnModule(X, torch.randn(16, d, generator=g, device="cuda"), torch.randn(d, 16, generator=g, device="cuda"))
    mod.sp_ffn_init()
    mod.sp_ffn_cache_input_inverse(0.1)
    G = mod.G_X.double()
    want = torch.linalg.inv(G + 0.1 * G.diagonal().mean() * torch.eye(d, device="cuda", dtype=torch.float64))
    assert float((mod.G_X_inv.double() - want).abs().max() / want.abs().max()) < 1.2e-7
    assert torch.equal(mod.G_X_inv, mod.G_X_inv.T)
    mod.check_status()


def _own_stream_calls(api, seed):
    """The calls that use the caller's stream alone, each as (call, its output)."""
    n, m = 200, 90
    g = torch.Generator(device="cuda").manual_seed(seed)
    G, R = _spd(n, seed), torch.randn(m, n, generator=g, device="cuda")
    mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    mask[::2] = 1
    mod = api.FfnModule(torch.randn(2 * n, n, generator=g, device="cuda").bfloat16(),
                        torch.randn(16, n, generator=g, device="cuda"), torch.randn(n, 16, generator=g, device="cuda"))
    mod.sp_ffn_init()
    mod.G_X_inv = torch.zeros(n, n, device="cuda")
    ws = [torch.empty(api.workspace_bytes(op, m, n, 0, 0, api.SP_F64), dtype=torch.uint8, device="cuda") for op in (7, 5)]
    W = [torch.zeros(m, n, device="cuda") for _ in range(2)]
    return {"solve": (lambda: api.sp_ridge_solve(R, G, 0.1, True, precise=True, W=W[0], ws=ws[0]), W[0]),
            "refit": (lambda: api.sp_linear_refit(R, G, mask, n // 2, 0.1, precise=True, W=W[1], ws=ws[1]), W[1]),
            "inverse": (lambda: mod.sp_ffn_cache_input_inverse(0.1), mod.G_X_inv)}


@pytest.mark.parametrize("name", ["solve", "refit", "inverse"])
def test_calls_on_the_callers_stream_alone_beside_a_capture(name):
    """Issued on a stream of its own while another stream's capture holds the library's assisting streams: neither the call
    nor the capture fails, and the call itself can be captured."""
    api = _api()
    call, out = _own_stream_calls(api, 3)[name]
    call()
    torch.cuda.synchronize()
    want = out.clone()
    G, R = _spd(600, 5), torch.randn(64, 600, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    W = torch.zeros_like(R)
    ws = torch.empty(api.workspace_bytes(7, 64, 600, 0, 0, api.SP_F32), dtype=torch.uint8, device="cuda")
    forks = lambda: api.sp_ridge_solve(R, G, 0.1, True, W=W, ws=ws)
    api.sp_set_reproducible(True)
    try:
        forks()
        torch.cuda.synchronize()
        want_W = W.clone()
        cap, other = torch.cuda.Stream(), torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=cap, capture_error_mode="relaxed"):
            forks()
            with torch.cuda.stream(other):
                out.zero_()
                call()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        W.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(W, want_W)
    finally:
        api.sp_set_reproducible(False)
    own = torch.cuda.CUDAGraph()
    with torch.cuda.graph(own, stream=cap, capture_error_mode="relaxed"):
        call()
    for _ in range(2):
        out.zero_()
        own.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)


def test_calls_on_the_callers_stream_alone_from_several_threads():
    """Three host threads, each on a stream and buffers of its own."""
    import threading
    api = _api()
    jobs = [list(_own_stream_calls(api, seed).values()) for seed in (11, 12, 13)]
    for job in jobs:
        for call, _ in job:
            call()
    torch.cuda.synchronize()
    want = [[out.clone() for _, out in job] for job in jobs]
    got = [[] for _ in jobs]
    start = threading.Barrier(len(jobs))

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            for _ in range(8):
                for call, out in jobs[k]:
                    out.zero_()
                    call()
                got[k].append([out.clone() for _, out in jobs[k]])
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for k in range(len(jobs)):
        assert len(got[k]) == 8 and all(torch.equal(a, b) for r in got[k] for a, b in zip(r, want[k]))


@pytest.mark.parametrize("n", [1, 2, 3, 8, 31, 33, 64, 100, 128, 200, 255, 257, 520])
@pytest.mark.parametrize("precise", [False, True])
def test_refit_of_narrow_matrices(n, precise):
    """Right-hand sides of few columns: the kernels that gather, clear and scatter them put several rows into a block."""
    api = _api()
    m, k = 1237, (n + 1) // 2
    g = torch.Generator(device="cuda").manual_seed(n)
    G, R = _spd(n, n), torch.randn(m, n, generator=g, device="cuda")
    keep = torch.sort(torch.randperm(n, generator=g, device="cuda")[:k]).values
    mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    mask[keep] = 1
    W = torch.full((m + 1, n + 3), 7.0, device="cuda")
    api.sp_linear_refit(R, G, mask, k, 0.1, precise=precise, W=W[:m, :n], rho_relative=True)
    H = G[keep][:, keep].double() + 0.1 * G.double().diagonal().mean() * torch.eye(k, device="cuda", dtype=torch.float64)
    want = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    want[:, keep] = torch.linalg.solve(H, R[:, keep].double().T).T
    # fp64: rounded to fp32 once; fp32: a few 2^-24 times the condition number (the ridge bounds it by 10 n)
    bound = 1.2e-7 if precise else 4 * 2.0 ** -24 * 10 * max(n, 10)
    assert float((W[:m, :n].double() - want).abs().max() / want.abs().max()) < bound
    assert bool((W[:m, :n][:, mask == 0] == 0).all()) and bool((W[m] == 7).all()) and bool((W[:, n:] == 7).all())
