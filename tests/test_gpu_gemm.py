"""The three contractions of a layer in isolation (through lp_gemm_bf16) against their
definition, C = A.B in float64 on the same bf16 operands.  Sizes span several 128-wide
tiles with ragged tails, single-tile cases, and the degenerate small extents of the
workloads (N = 10, K = 784, M = 32)."""
import numpy as np
import pytest

from gpu_common import rel_l2

pytestmark = pytest.mark.gpu

SHAPES = [(128, 128, 64), (256, 384, 512), (32, 10, 784), (300, 200, 520), (1, 8, 8), (129, 65, 72),
          (512, 1000, 256), (64, 2056, 136)]


def _operands(which, M, N, K, seed):
    import torch
    g = torch.Generator(device="cpu").manual_seed(seed)
    pad8 = lambda v: (v + 7) // 8 * 8
    if which == 0:
        A = torch.randn(M, pad8(K), generator=g)
        B = torch.randn(N, pad8(K), generator=g)
    elif which == 1:
        A = torch.randn(M, pad8(K), generator=g)
        B = torch.randn(K, pad8(N), generator=g)
    else:
        A = torch.randn(K, pad8(M), generator=g)
        B = torch.randn(K, pad8(N), generator=g)
    return A.bfloat16(), B.bfloat16()


def _reference(which, M, N, K, A, B):
    a = A.double().numpy()
    b = B.double().numpy()
    if which == 0:
        return a[:, :K] @ b[:, :K].T
    if which == 1:
        return a[:, :K] @ b[:K, :N]
    return a[:K, :M].T @ b[:K, :N]


@pytest.mark.parametrize("tile_n", [0, 64, 256, 512, 448])      # 512 / 448 = 256 x 256 / 256 x 224 tile on an SM pair (cta_group::2)
@pytest.mark.parametrize("which", [0, 1, 2])
def test_contraction_matches_definition(which, tile_n):
    import torch
    from paper_2108_06629_b200 import binding as lpb
    lpb.lp_set_tuning(tile_n, 0)
    try:
        for i, (M, N, K) in enumerate(SHAPES):
            A, B = _operands(which, M, N, K, 100 * which + i)
            ref = _reference(which, M, N, K, A, B)
            ldc = (N + 3) // 4 * 4
            Cd = torch.full((M, ldc), 7.0, device="cuda")
            lpb.lp_gemm_bf16(which, M, N, K, A.cuda(), A.shape[1], B.cuda(), B.shape[1], Cd, ldc)
            torch.cuda.synchronize()
            got = Cd.cpu().numpy()
            assert rel_l2(got[:, :N], ref) < 1e-6 + 2e-7 * np.sqrt(K), (which, M, N, K)   # fp32 accumulation over K terms
            assert np.all(got[:, N:] == 0.0)          # pad lanes of the last 16-byte group are zeroed
    finally:
        lpb.lp_set_tuning(0, 0)


def test_deep_pipeline_and_two_stage_pipeline_agree():
    import torch
    from paper_2108_06629_b200 import binding as lpb
    M, N, K = 256, 256, 4096
    A, B = _operands(0, M, N, K, 7)
    outs = []
    for stages in (2, 6):
        lpb.lp_set_tuning(128, stages)
        Cd = torch.empty((M, N), device="cuda")
        lpb.lp_gemm_bf16(0, M, N, K, A.cuda(), K, B.cuda(), K, Cd, N)
        torch.cuda.synchronize()
        outs.append(Cd.cpu().numpy())
    lpb.lp_set_tuning(0, 0)
    assert np.array_equal(outs[0], outs[1])
    assert rel_l2(outs[0], _reference(0, M, N, K, A, B)) < 1e-6 + 2e-7 * np.sqrt(K)


def test_status_word_is_clear_after_ordinary_launches():
    import torch
    from paper_2108_06629_b200 import binding as lpb
    A, B = _operands(0, 256, 384, 512, 3)
    Cd = torch.empty((256, 384), device="cuda")
    lpb.lp_gemm_bf16(0, 256, 384, 512, A.cuda(), 512, B.cuda(), 512, Cd, 384)
    rc, word = lpb.lp_gemm_status()
    assert (rc, word) == (lpb.LP_OK, 0)


def test_bounded_wait_runs_out_reports_and_leaves_the_device_usable():
    """Every barrier wait in the kernels is bounded.  Here one is made to run out in the harmless
    way the library offers for it: the producer skips the last k-block, the MMA issuer waits for it
    for 2e6 cycles (about a millisecond) and gives up.  The kernel must return by itself, the
    status word must say so, and the next ordinary launch must be exact and leave the word clear."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    M, N, K = 256, 384, 512
    A, B = _operands(0, M, N, K, 11)
    Ad, Bd = A.cuda(), B.cuda()
    Cd = torch.zeros((M, N), device="cuda")
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    lpb.lp_debug_gemm_starved(M, N, K, Ad, K, Bd, K, Cd, N, 2_000_000)
    t1.record()
    rc, word = lpb.lp_gemm_status()            # waits for the device
    assert rc == lpb.LP_ERR_TIMEOUT and word in (2, 3), (rc, word)
    assert b"bounded" in lpb.lib().lp_last_error(None)
    assert t0.elapsed_time(t1) < 500.0         # gave up after the short limit, not after seconds
    # what did arrive was contracted: the result is the product over the first K - 64 columns (if the
    # epilogue's own wait had not run out first, in which case C was left alone)
    if word == 2:
        ref = A.double().numpy()[:, :K - 64] @ B.double().numpy()[:, :K - 64].T
        assert rel_l2(Cd.cpu().numpy(), ref) < 1e-5
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)          # reading the word cleared it
    lpb.lp_gemm_bf16(0, M, N, K, Ad, K, Bd, K, Cd, N)
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)
    assert rel_l2(Cd.cpu().numpy(), _reference(0, M, N, K, A, B)) < 1e-6 + 2e-7 * np.sqrt(K)
    # argument checks of the verification call
    lib = lpb.lib()
    assert lib.lp_debug_gemm_starved(M, N, 64, None, K, None, K, None, N, 2_000_000, None) == lpb.LP_ERR_INVALID_ARG
    assert lib.lp_debug_gemm_starved(M, N, K, Ad.data_ptr(), K, Bd.data_ptr(), K, Cd.data_ptr(), N, 5, None) == lpb.LP_ERR_INVALID_ARG


# Outputs of few tiles, where the contraction is divided over a cluster: as many and more k-blocks than CTAs, ranks with
# one k-block more than others, a ragged last k-block, clusters of 2, 4 and 8, tiles of 64 and 128 columns with ragged edges, one row.
CLUSTER_SHAPES = [(1, 8, 65), (33, 70, 128), (128, 64, 200), (100, 777, 1003), (129, 130, 256), (64, 2050, 4100), (250, 513, 1000),
                  (40, 300, 4160), (384, 1000, 3000), (300, 4100, 1100), (300, 4100, 2100)]


@pytest.mark.parametrize("which", [0, 1, 2])
def test_contraction_divided_over_a_cluster(which):
    """Against float64; the partial sums are shorter than the undivided one, so its bound holds."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    forms = set()
    for i, (M, N, K) in enumerate(CLUSTER_SHAPES):
        A, B = _operands(which, M, N, K, 900 + 100 * which + i)
        ldc = (N + 3) // 4 * 4
        Cd = torch.full((M, ldc), 7.0, device="cuda")
        Ad, Bd = A.cuda(), B.cuda()
        lpb.lp_gemm_bf16(which, M, N, K, Ad, A.shape[1], Bd, B.shape[1], Cd, ldc)
        forms.add(lpb.lp_debug_last_contraction())
        torch.cuda.synchronize()
        got = Cd.cpu().numpy()
        assert rel_l2(got[:, :N], _reference(which, M, N, K, A, B)) < 1e-6 + 2e-7 * np.sqrt(K), (which, M, N, K)
        assert np.all(got[:, N:] == 0.0)
        assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)
    assert {"cluster 64 x2", "cluster 64 x4", "cluster 64 x8", "cluster 128 x2"} <= forms, forms


def _sum_of_parts(which, M, N, A, B, ldc, k0, k1, parts):
    """The product over [k0, k1) as undivided contractions of consecutive k-blocks, added in order: parts[0] of them (the first ones
    a k-block longer), each made in turn of parts[1] of them, ..."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    if not parts:
        C = torch.zeros((M, ldc), device="cuda")
        a = A[k0:k1] if which == 2 else A[:, k0:k1]
        b = B[:, k0:k1] if which == 0 else B[k0:k1]
        lpb.lp_set_tuning(64, 0, 1)                  # (64-column tiles, one CTA each)
        try:
            lpb.lp_gemm_bf16(which, M, N, k1 - k0, a, A.shape[1], b, B.shape[1], C, ldc)
        finally:
            lpb.lp_set_tuning(0, 0, 0)
        assert lpb.lp_debug_last_contraction().startswith("single 64")
        return C
    kb, total = (k1 - k0 + 63) // 64, None
    for r in range(parts[0]):
        end = min(k1, k0 + 64 * (kb // parts[0] + (r < kb % parts[0])))
        C = _sum_of_parts(which, M, N, A, B, ldc, k0, end, parts[1:])
        total = C if total is None else total + C
        k0 = end
    return total


# CTAs of a cluster, accumulators of a CTA: one to four k-blocks on tiles that leave room for four CTAs, for two and for one; 75 and more
# tiles on both sides of 32 k-blocks; 74 tiles (halves) on both sides of 64.
@pytest.mark.parametrize("M, N, K, parts", [
    (64, 64, 256, (1, 4)), (33, 70, 250, (1, 4)), (128, 2368, 200, (1, 4)), (128, 2369, 200, (1, 2)), (129, 65, 130, (1, 2)), (1, 1, 128, (1, 2)),
    (300, 1000, 256, (1, 2)), (513, 1000, 256, (1, 1)), (65, 130, 40, (1, 1)), (1000, 1000, 2100, (1, 2)), (128, 4800, 1980, (1, 1)),
    (120, 6008, 4040, (1, 2)), (64, 4736, 4096, (2, 2)), (100, 4730, 4290, (2, 2)), (64, 4736, 4030, (2, 1))])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_sums_of_a_contraction_are_no_longer_than_its_parts(which, M, N, K, parts):
    """The accumulator is truncated once per 16 terms, so its error grows with the length of a sum: bit for bit the sums of
    the parts, added in order."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    A, B = (t.cuda() for t in _operands(which, M, N, K, 5000 + which))
    ldc = (N + 3) // 4 * 4
    Cd = torch.full((M, ldc), 7.0, device="cuda")
    lpb.lp_gemm_bf16(which, M, N, K, A, A.shape[1], B, B.shape[1], Cd, ldc)
    assert lpb.lp_debug_last_contraction() == "cluster 64 x%d" % parts[0]
    assert torch.equal(Cd, _sum_of_parts(which, M, N, A, B, ldc, 0, K, parts))
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)


# Two CTAs an SM: one and several rows of tiles, the most tiles of quarters and the fewest and most of halves, k-blocks on the line and an odd
# number of them; and the same where a row, or the matrix, does not start on a sector (shift: elements).
@pytest.mark.parametrize("M, N, K, shift, parts", [
    (64, 4096, 4096, 0, (4,)), (256, 2048, 4096, 0, (4,)), (384, 1024, 4096, 0, (4,)), (112, 2448, 4144, 0, (4,)), (64, 4352, 4096, 0, (4,)),
    (64, 4736, 4096, 0, (2, 2)), (64, 2416, 4032, 0, (2,)), (64, 4752, 2048, 0, (2,)), (1008, 1152, 2064, 0, (2,)), (1008, 1152, 1984, 0, (1,)),
    (120, 2504, 4104, 0, (2, 2)), (120, 6008, 2056, 0, (1, 2)), (64, 4096, 4096, 8, (2, 2)), (1008, 1152, 2064, 8, (1, 2))])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_long_contraction_is_divided_over_two_ctas_an_sm(which, M, N, K, shift, parts):
    """The form, and bit for bit the sums of its parts."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    A, B = (t.cuda() for t in _operands(which, M, N, K, 4000 + which))
    if shift:
        B = torch.nn.functional.pad(B.reshape(-1), (shift, 0))[shift:].view(B.shape)
    ldc = (N + 3) // 4 * 4
    Cd = torch.full((M, ldc), 7.0, device="cuda")
    lpb.lp_gemm_bf16(which, M, N, K, A, A.shape[1], B, B.shape[1], Cd, ldc)
    assert lpb.lp_debug_last_contraction() == "cluster 64 x%d" % parts[0]
    assert torch.equal(Cd, _sum_of_parts(which, M, N, A, B, ldc, 0, K, parts))
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)


# Plain fp32 results on SM pairs: at least two tiles a pair (persistent, 256 and 224 columns, MN-major A in the G form), and no
# more tiles than pairs (six stages), with ragged last rows, columns and k-blocks.
@pytest.mark.parametrize("which, M, N, K, form", [
    (0, 1024, 9467, 1100, "pair persistent 256"), (1, 1024, 9467, 1100, "pair persistent 256"), (2, 1024, 9467, 1100, "pair persistent 256"),
    (0, 1100, 7677, 1030, "pair persistent 224"), (1, 1100, 7677, 1030, "pair persistent 224"), (2, 1100, 7677, 1030, "pair persistent 256"),
    (0, 1030, 1100, 1040, "pair 224 x6"), (1, 1030, 1100, 1040, "pair 224 x6"), (2, 1030, 1100, 1040, "pair 256 x6")])
def test_contraction_on_sm_pairs(which, M, N, K, form):
    import torch
    from paper_2108_06629_b200 import binding as lpb
    A, B = _operands(which, M, N, K, 77 + which)
    ldc = (N + 3) // 4 * 4
    Cd = torch.full((M, ldc), 7.0, device="cuda")
    lpb.lp_gemm_bf16(which, M, N, K, A.cuda(), A.shape[1], B.cuda(), B.shape[1], Cd, ldc)
    assert lpb.lp_debug_last_contraction() == form
    torch.cuda.synchronize()
    got = Cd.cpu().numpy()
    assert rel_l2(got[:, :N], _reference(which, M, N, K, A, B)) < 1e-6 + 2e-7 * np.sqrt(K)
    assert np.all(got[:, N:] == 0.0)
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)


@pytest.mark.parametrize("B, n, classes", [(33, 200, 10), (128, 1000, 513), (300, 64, 1000)])
def test_kernels_of_a_stream_see_what_the_one_before_wrote(B, n, classes):
    """Launches of one stream start before the kernel in front of them has ended and wait inside.  A chain in which every
    call reads what the call before it wrote (loss -> contraction -> loss ...), enqueued at once, against the same with the
    device idle between the calls, and captured into a graph that is replayed: bit for bit."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    g = torch.Generator().manual_seed(B)
    ld, ldc = (n + 7) // 8 * 8, (classes + 7) // 8 * 8
    w = torch.zeros(classes, ld, dtype=torch.bfloat16)
    w[:, :n] = torch.randn(classes, n, generator=g) * n ** -0.5
    w = w.cuda()
    y = torch.randint(0, classes, (B,), generator=g, dtype=torch.int32).cuda()
    z0 = torch.randn(B, ldc, generator=g).cuda()

    def chain(wait):
        z, e = z0.clone(), torch.zeros(B, ld, device="cuda")
        d, loss, dw = torch.zeros(B, ldc, dtype=torch.bfloat16, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros(classes, ld, device="cuda")
        a = torch.zeros(B, ld, dtype=torch.bfloat16, device="cuda")

        def once():
            for _ in range(6):
                assert lpb.lp_softmax_xent_static(z, y, d, loss, classes) == lpb.LP_OK
                wait()
                lpb.lp_gemm_bf16(1, B, n, classes, d, ldc, w, ld, e, ld)
                wait()
                a.copy_(e * B)
                wait()
                lpb.lp_gemm_bf16(2, classes, n, B, d, ldc, a, ld, dw, ld)
                wait()
                lpb.lp_gemm_bf16(0, B, classes, n, a, ld, w, ld, z, ldc)
                wait()
        return once, (z, e, d, loss, dw)

    once, want = chain(torch.cuda.synchronize)
    once()
    for _ in range(3):
        once, got = chain(lambda: None)
        once()
        torch.cuda.synchronize()
        assert all(torch.equal(p, q) for p, q in zip(want, got))
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    once, got = chain(lambda: None)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        once()
    got[0].copy_(z0)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(p, q) for p, q in zip(want, got))


@pytest.mark.parametrize("which", [0, 1, 2])
def test_undivided_contraction_in_the_cluster_form(which):
    """A cluster of one: one to four k-blocks with ragged ends, one element, ragged tiles, the most tiles, and long contractions
    of tiles that fill the SMs by themselves."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    for i, (M, N, K) in enumerate([(1, 1, 1), (33, 70, 10), (129, 65, 250), (513, 1000, 256), (128, 9400, 60), (800, 1300, 700), (1000, 1000, 2100)]):
        A, B = _operands(which, M, N, K, 3000 + 100 * which + i)
        ldc = (N + 3) // 4 * 4
        Cd = torch.full((M, ldc), 7.0, device="cuda")
        lpb.lp_gemm_bf16(which, M, N, K, A.cuda(), A.shape[1], B.cuda(), B.shape[1], Cd, ldc)
        assert lpb.lp_debug_last_contraction() == "cluster 64 x1", (M, N, K)
        torch.cuda.synchronize()
        got = Cd.cpu().numpy()
        assert rel_l2(got[:, :N], _reference(which, M, N, K, A, B)) < 1e-6 + 2e-7 * np.sqrt(K), (which, M, N, K)
        assert np.all(got[:, N:] == 0.0)
    assert lpb.lp_gemm_status() == (lpb.LP_OK, 0)
