"""lp_softmax_xent_static: the loss kernel for callers that have no workspace to offer and
may not allocate one (see the header).  Its scratch is a fixed array inside the library,
so this test checks what such a caller relies on: the results equal those of the loss task
run through a trainer handle on the same logits and labels, on two calls in a row (the
second call finds the first call's leftovers in the shared scratch), and oversize batches
are refused without launching anything.

Collected last on purpose (file name): a failure here cannot mask any other test."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _through_handle(tr, n, logits, labels):
    tr.debug_write("logits", 0, n, logits)
    tr.debug_write("labels", 0, n, labels.astype(np.float32))
    tr.debug_run_task("loss", 0, n)
    L = len(tr.layers)
    return tr.debug_read("delta", L - 1, n), float(tr.debug_read("loss", 0, n)[0])


def test_static_scratch_loss_matches_handle_loss_twice_in_a_row():
    import torch
    from paper_2108_06629_b200 import binding as lpb
    from paper_2108_06629_b200 import inputs as I

    batch, classes = 200, 1003                     # ragged: 1003 is not a multiple of 8
    layers = I.mlp([64, classes], "relu")
    W0, b0 = I.initial_weights(layers, 0)
    tr = lpb.Trainer(layers, batch, 1, W0=W0, b0=b0)
    ld = (classes + 7) // 8 * 8
    rng = np.random.default_rng(77)
    for call in range(2):                          # two calls in a row on the shared scratch
        logits = (rng.standard_normal((batch, classes)) * (3.0 + 5.0 * call)).astype(np.float32)
        labels = rng.integers(0, classes, size=batch).astype(np.int32)
        want_delta, want_loss = _through_handle(tr, call, logits, labels)

        lg = torch.zeros((batch, ld), dtype=torch.float32, device="cuda")
        lg[:, :classes] = torch.from_numpy(logits).cuda()
        lb = torch.from_numpy(labels).cuda()
        delta = torch.full((batch, ld), 7.0, dtype=torch.bfloat16, device="cuda")
        loss = torch.full((1,), -1.0, dtype=torch.float32, device="cuda")
        rc = lpb.lp_softmax_xent_static(lg, lb, delta, loss, classes)
        assert rc == lpb.LP_OK
        torch.cuda.synchronize()
        got_delta = delta.float().cpu().numpy()
        # same kernel, same inputs: bf16 results must agree to the bit, the loss to fp32 round-off
        assert np.array_equal(got_delta[:, :classes], want_delta)
        assert np.all(got_delta[:, classes:] == 0.0)
        assert abs(float(loss.item()) - want_loss) <= 1e-6 * max(1.0, abs(want_loss))
        # and the loss is what its definition says (float64, from the same logits)
        z = logits.astype(np.float64)
        lse = np.log(np.exp(z - z.max(1, keepdims=True)).sum(1)) + z.max(1)
        assert abs(float(loss.item()) - float(np.mean(lse - z[np.arange(batch), labels]))) < 1e-4
    tr.close()


def test_static_scratch_loss_refuses_what_does_not_fit():
    import torch
    from paper_2108_06629_b200 import binding as lpb
    big = lpb.LP_XENT_STATIC_MAX_BATCH + 1
    lg = torch.zeros((big, 8), dtype=torch.float32, device="cuda")
    lb = torch.zeros((big,), dtype=torch.int32, device="cuda")
    delta = torch.full((big, 8), 7.0, dtype=torch.bfloat16, device="cuda")
    loss = torch.full((1,), -1.0, dtype=torch.float32, device="cuda")
    assert lpb.lp_softmax_xent_static(lg, lb, delta, loss, 8) == lpb.LP_ERR_INVALID_ARG
    torch.cuda.synchronize()
    assert float(loss.item()) == -1.0 and float(delta.float().min().item()) == 7.0     # nothing ran
    # pitch too small for the padded row, and the largest batch that does fit
    narrow = torch.zeros((16, 4), dtype=torch.bfloat16, device="cuda")
    assert lpb.lp_softmax_xent_static(lg[:16], lb[:16], narrow, loss, 8) == lpb.LP_ERR_INVALID_ARG
    ok = lpb.LP_XENT_STATIC_MAX_BATCH
    assert lpb.lp_softmax_xent_static(lg[:ok], lb[:ok], delta[:ok], loss, 8) == lpb.LP_OK
    torch.cuda.synchronize()
    # all-zero logits: uniform softmax, loss = log 8 (16384 row losses added in fp32)
    assert abs(float(loss.item()) - np.log(8.0)) < 1e-3 * np.log(8.0)
    # the refusals say why
    assert lpb.lp_softmax_xent_static(lg, lb, delta, loss, 8) == lpb.LP_ERR_INVALID_ARG
    assert b"LP_XENT_STATIC_MAX_BATCH" in lpb.lib().lp_last_error(None)


def test_static_scratch_loss_never_uses_a_bad_label_as_an_address():
    """This entry point has no status word to report through, so a label outside [0, classes)
    shows up as a NaN loss; the rows with valid labels are unaffected and nothing faults."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    batch, classes = 16, 8
    lg = torch.zeros((batch, classes), dtype=torch.float32, device="cuda")
    delta = torch.zeros((batch, classes), dtype=torch.bfloat16, device="cuda")
    loss = torch.zeros((1,), dtype=torch.float32, device="cuda")
    for bad in (8, -1, 2 ** 31 - 1):
        lb = torch.zeros((batch,), dtype=torch.int32, device="cuda")
        lb[5] = bad
        assert lpb.lp_softmax_xent_static(lg, lb, delta, loss, classes) == lpb.LP_OK
        torch.cuda.synchronize()
        assert np.isnan(float(loss.item()))
        d = delta.float().cpu().numpy()
        assert abs(d[0, 0] - (1.0 / 8 - 1.0) / batch) < 1e-3 and abs(d[5, 0] - (1.0 / 8) / batch) < 1e-3
    lb = torch.zeros((batch,), dtype=torch.int32, device="cuda")
    assert lpb.lp_softmax_xent_static(lg, lb, delta, loss, classes) == lpb.LP_OK
    torch.cuda.synchronize()
    assert abs(float(loss.item()) - np.log(8.0)) < 1e-5


@pytest.mark.parametrize("B, C, ld", [(1, 1, 1), (3, 2, 2), (9, 1000, 1000), (7, 1001, 1003), (8, 1024, 1024), (5, 1025, 1026),
                                      (4, 8192, 8192), (3, 8195, 8195), (300, 33, 40),
                                      # eight threads a row: one class, 64 and 65, rows that end inside a warp; four classes an access and a ragged last four;
                                      # more rows than a pass of the grid; 257, 2048 and 2049 classes
                                      (67, 1, 4), (133, 64, 64), (70, 65, 68), (131, 61, 64), (16384, 10, 12), (9500, 258, 260),
                                      (33, 257, 257), (41, 2048, 2048), (40, 2049, 2052), (37, 2047, 2048)])
def test_static_loss_at_the_edges_of_its_row_forms(B, C, ld):
    """A warp or a block per row, classes beyond what the registers hold, odd pitches (one class per access), a masked
    class (-inf logit): loss and delta against float64.  One bf16 rounding of delta; fp32 sums over C classes."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    g = torch.Generator().manual_seed(B * 10007 + C)
    z = torch.full((B, ld), 1e30)
    z[:, :C] = 3.0 * torch.randn(B, C, generator=g)
    y = torch.randint(0, C, (B,), generator=g, dtype=torch.int32)
    if C > 2:
        z[0, (int(y[0]) + 1) % C] = float("-inf")
    ldd = (C + 7) // 8 * 8 + (ld % 2)
    delta = torch.full((B, ldd), 7.0, dtype=torch.bfloat16, device="cuda")
    loss = torch.zeros(1, device="cuda")
    for _ in range(2):
        assert lpb.lp_softmax_xent_static(z.cuda(), y.cuda(), delta, loss, C) == lpb.LP_OK
    logp = torch.log_softmax(z[:, :C].double(), 1)
    rows = torch.arange(B)
    want = logp.exp()
    want[rows, y.long()] -= 1.0
    want /= B
    ref_loss = float(-logp[rows, y.long()].mean())
    got = delta.double().cpu()
    assert torch.all((got[:, :C] - want).abs() <= 2.0 ** -8 * want.abs() + 1e-6 / B)
    assert torch.all(got[:, C:(C + 7) // 8 * 8] == 0.0)
    assert abs(float(loss) - ref_loss) <= 2e-6 * max(1.0, abs(ref_loss))


@pytest.mark.parametrize("B, C", [(1, 10), (64, 10), (300, 10), (3000, 10), (1025, 100), (2049, 1000), (700, 1100), (16384, 33)])
def test_static_loss_is_the_loss_task_bit_for_bit(B, C):
    """The same logits through a trainer's loss task and through the static call: one block, a few, more rows than sums."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    from paper_2108_06629_b200 import inputs as I
    g = torch.Generator().manual_seed(B + C)
    z = torch.zeros(B, (C + 7) // 8 * 8)
    z[:, :C] = 3.0 * torch.randn(B, C, generator=g)
    y = torch.randint(0, C, (B,), generator=g, dtype=torch.int32)
    layers = [I.fc(8, C, "none")]
    W0, b0 = I.initial_weights(layers, 0)
    tr = lpb.Trainer(layers, B, 1, W0=W0, b0=b0)
    tr.debug_write("labels", 0, 0, y.float().numpy())
    tr.debug_write("logits", 0, 0, z[:, :C].numpy())
    tr.debug_run_task("loss", 0, 0)
    delta, loss = torch.zeros(B, z.shape[1], dtype=torch.bfloat16, device="cuda"), torch.zeros(1, device="cuda")
    assert lpb.lp_softmax_xent_static(z.cuda(), y.cuda(), delta, loss, C) == lpb.LP_OK
    assert np.array_equal(tr.debug_read("delta", 0, 0), delta[:, :C].float().cpu().numpy())
    assert float(tr.debug_read("loss", 0, 0)[0]) == float(loss)
    tr.close()


def test_static_loss_after_calls_that_overlapped():
    """Two calls that overlap on the shared scratch may give wrong losses and leave its counter anywhere; the header
    promises that ordered calls after them are right again.  16 pairs of calls of many blocks, numbers unequal, run on
    two streams at the same time; then ordered calls of many batch sizes against float64."""
    import torch
    from paper_2108_06629_b200 import binding as lpb
    C, wide, big = 1000, 4000, [3000, 2900]
    g = torch.Generator().manual_seed(3)
    z = torch.randn(8192, C, generator=g)
    y = torch.randint(0, C, (8192,), generator=g, dtype=torch.int32)
    zd, yd, zw = z.cuda(), y.cuda(), torch.randn(3000, wide, device="cuda")
    delta, loss = torch.zeros(8192, C, dtype=torch.bfloat16, device="cuda"), torch.zeros(1, device="cuda")
    scrap = [torch.zeros(3000, wide, dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    losses = [torch.zeros(1, device="cuda") for _ in range(3)]
    streams, hold = [torch.cuda.Stream() for _ in range(2)], torch.cuda.Stream()
    for _ in range(16):
        torch.cuda.synchronize()
        with torch.cuda.stream(hold):
            torch.cuda._sleep(20_000_000)             # (about ten milliseconds: both calls are enqueued before it ends)
            gate = hold.record_event()
        for k, s in enumerate(streams):
            s.wait_event(gate)
            with torch.cuda.stream(s):
                assert lpb.lp_softmax_xent_static(zw[:big[k]], yd[:big[k]], scrap[k], losses[k], wide) == lpb.LP_OK
            for _ in range(63 if k == 0 else 0):      # (counters may be handed out in turn: the pair shares one of 64)
                assert lpb.lp_softmax_xent_static(zw, yd[:3000], scrap[2], losses[2], wide) == lpb.LP_OK
    torch.cuda.synchronize()
    logp = torch.log_softmax(z.double(), 1)
    for i in range(130):
        B = 2048 + 47 * i
        labels = (y[:B] + 7 * i) % C                  # (new row losses: what the scratch holds from the call before is wrong)
        assert lpb.lp_softmax_xent_static(zd[:B], labels.cuda(), delta, loss, C) == lpb.LP_OK
        want = float(-logp[torch.arange(B), labels.long()].mean())
        assert abs(float(loss) - want) <= 2e-6 * max(1.0, abs(want)), (i, B)
