"""The error contract of the C ABI on a device: the status word a kernel's bounded wait writes, what
d2c_sync_status reports from it, and the argument checks that need a live context."""
import contextlib
import ctypes
import mmap
from dataclasses import replace

import pytest
import torch

from paper_2509_23094_b200 import binding, inputs
from gpu_util import Pair

pytestmark = pytest.mark.gpu


def test_status_word_is_reported_and_sticky_until_cleared():
    wl = inputs.WORKLOADS["toy"]
    pair = Pair(wl)
    pair.gpu_step(10 ** 6, 1.0)                                     # a clean step: status stays 0
    st = pair.ctx.view("status")
    assert st.tolist() == [0, 0, 0, 0]
    # what a kernel's wait that ran out leaves behind: the code and the number of the wait
    st.copy_(torch.tensor([binding.D2C_ETIMEOUT, 32, 0, 0], dtype=torch.int32))
    with pytest.raises(binding.D2cError) as e:
        pair.ctx.sync_status()
    assert e.value.code == binding.D2C_ETIMEOUT and "site 32" in str(e.value)
    with pytest.raises(binding.D2cError):                           # sticky: still there on the next call
        pair.ctx.sync_status()
    st.zero_()
    pair.ctx.sync_status()
    g = pair.gpu_step(wl.k, wl.p)                                   # and the context is as usable as before
    assert 0 < len(g["sel"][0]) < wl.seq_len


def test_a_bounded_wait_that_runs_out_returns_and_records_the_timeout():
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    binding.d2c_op_wait_probe(status, limit_cycles=100000)          # ~50 us: nothing ever arrives on the barrier
    torch.cuda.synchronize()                                        # the kernel came back by itself
    assert status.tolist()[:2] == [binding.D2C_ETIMEOUT, 99]
    # the first error wins: a second run does not overwrite the site
    status[1] = 7
    binding.d2c_op_wait_probe(status, limit_cycles=50000)
    torch.cuda.synchronize()
    assert status.tolist()[:2] == [binding.D2C_ETIMEOUT, 7]
    # the device is fine afterwards
    x = torch.arange(8, device="cuda").sum().item()
    assert x == 28
    with pytest.raises(binding.D2cError):
        binding.d2c_op_wait_probe(status, limit_cycles=10)          # limits outside [1e3, 2e9] are refused on the host


def test_threads_that_meet_leave_together_when_a_wait_gives_up():
    """Another warp's wait runs out while 256 threads go from one named barrier to the next: whenever the flag is set, all of
    them leave at the same one (a thread that stayed would wait there for good)."""
    for limit in (1000, 1234, 5000, 20011, 100003, 1000003):
        for _ in range(20):
            status = torch.zeros(4, dtype=torch.int32, device="cuda")
            binding.d2c_op_wait_probe(status, limit_cycles=limit)
            assert status.tolist() == [binding.D2C_ETIMEOUT, 99, 256, 0]


def test_a_context_keeps_the_batch_and_length_of_its_first_step():
    wl = inputs.WORKLOADS["toy"]
    pair = Pair(wl, max_batch=2, max_seq=wl.seq_len + 64)
    pair.gpu_step(10 ** 6, 1.0)
    B, L, d = wl.batch, wl.seq_len, wl.shape.d_model
    h0 = torch.zeros(2, L, d, dtype=torch.bfloat16, device="cuda")
    mask = torch.ones(2, L, dtype=torch.uint8, device="cuda")
    with pytest.raises(binding.D2cError) as e:
        pair.ctx.step(h0, mask, 4, 0.5)                              # fits max_batch x max_seq, but is another layout
    assert e.value.code == binding.D2C_EINVAL and "first used" in str(e.value)
    with pytest.raises(binding.D2cError) as e:
        pair.ctx.step(h0[:1, : L - 8].contiguous(), mask[:1, : L - 8].contiguous(), 4, 0.5)
    assert e.value.code == binding.D2C_EINVAL
    g = pair.gpu_step(wl.k, wl.p)                                   # the original shape still works
    assert len(g["sel"][0]) > 0


def test_counts_left_by_a_wait_that_gave_up_do_not_reach_the_next_step():
    """A projection whose bounded wait ran out leaves the counters of its shared items as they are; a later launch that
    trusted them would add parts of another launch.  Every step starts with cleared ones: the same bits, whatever is there."""
    shape, seq = replace(inputs.TOY_HD128, name="deep", d_model=1024, d_ffn=2880, n_q_heads=8, n_kv_heads=8, vocab=4106), 701
    wl = inputs.Workload("deep", shape, 1, seq, 8, seq - 8, "all", 0, 0.0, seed=5)
    w = inputs.make_weights(shape, seed=5, device="cuda", gain_jitter=0.05)
    mask = inputs.make_mask(wl)
    h0, mask = inputs.make_h0(w["embed"].cpu(), inputs.make_tokens(wl, mask)).cuda(), mask.cuda()
    conf0 = inputs.make_scores(seq, 7).view(1, seq).cuda()
    ctx = binding.Context(binding.make_config(shape, 1, seq), w)
    # right before gemm_clocks: arrival and done counters of the one-SM kernel, and two sets of arrival counters of the pair kernel
    n = 2 * 320 + 2 * 160
    counters = ctx._view(ctx.state.gemm_clocks - 4 * n, n, torch.int32)
    sets = {"one-SM": counters[:640], "pair, first set": counters[640:800], "pair, second set": counters[800:]}
    hid = torch.zeros(seq, shape.d_model, dtype=torch.bfloat16, device="cuda")
    ctx.step(h0, mask, seq, 1.0)
    for rows in (257, 96):                                          # shared between clusters with many and with few rows
        runs = []
        for left in (None, 0, 1, 1000):
            if left is not None:
                counters.fill_(left)
            ctx.view("conf", 1, seq).copy_(conf0)
            hid.zero_()
            ctx.step(h0, mask, rows, 0.0, hidden_out=hid)
            ctx.sync_status()
            for name, part in sets.items():
                assert not part.any(), name
            runs.append([hid.clone(), ctx.view("kcache").clone(), ctx.view("conf").clone(), ctx.view("c").clone()])
        for other in runs[2:]:                                      # (the first step expects other rows than it finds)
            assert all(torch.equal(a, b) for a, b in zip(other, runs[1]))


def test_a_small_step_whose_grid_never_meets_has_no_rows_and_says_so():
    """A counter that starts far below what the CTAs of a one-launch step add to it: their first wait runs out (2 s), none of them takes an
    index from the memory that it waited for, so there are no rows and nothing of the state changes, the status tells, and the step behind
    it finds the counters at zero again."""
    wl = inputs.WORKLOADS["toy"]
    pair = Pair(wl)
    shape, seq, d = wl.shape, wl.seq_len, wl.shape.d_model
    hid, off = torch.zeros(seq, d, dtype=torch.bfloat16, device="cuda"), torch.full((2,), -1, dtype=torch.int32, device="cuda")
    h0, mask, scores = pair.h0.cuda(), pair.mask.cuda(), inputs.make_scores(seq, 8).view(1, seq).cuda()
    logits = torch.zeros(seq, shape.vocab, device="cuda")

    def step():
        pair.ctx.view("conf", 1, seq).copy_(scores)
        hid.zero_(); logits.zero_(); off.fill_(-1)
        pair.ctx.step(h0, mask, wl.k, 0.5, override_c=scores, hidden_out=hid, row_off=off, logits=logits)
        state = [pair.ctx.view(name).clone() for name in ("kcache", "vcache", "conf", "pred", "c")]
        return state + [hid.clone(), logits.clone(), off.clone()]

    pair.gpu_step(10 ** 6, 1.0)
    step()
    want = step()
    assert int(want[-1][1]) > wl.k
    count = pair.ctx._view(pair.ctx.state.status + 128, 2, torch.int32)       # arrivals of the grid's CTAs, and of those that leave
    assert count.tolist() == [0, 0]
    count[0] = -2 ** 30
    got = step()
    assert count.tolist() == [0, 0]
    with pytest.raises(binding.D2cError) as e:
        pair.ctx.sync_status()
    assert e.value.code == binding.D2C_ETIMEOUT and "site 60" in str(e.value)
    assert got[-1].tolist() == [0, 0] and not got[-2].any() and not got[-3].any()
    want_none = want[:2] + [scores] + want[3:5]                               # (of the step before; the confidences were put back since)
    assert all(torch.equal(a, b) for a, b in zip(got[:5], want_none))
    pair.ctx.view("status").zero_()
    assert all(torch.equal(a, b) for a, b in zip(step(), want))
    pair.ctx.sync_status()


def test_an_older_error_of_the_caller_is_not_taken_for_a_launch_error():
    """The thread's last CUDA error may be the caller's own, of a call that has nothing to do with the library."""
    def older():                                                    # refused, and remembered as the last error
        assert int(torch.cuda.cudart().cudaHostUnregister(torch.zeros(8).data_ptr())) != 0
    shape, seq = inputs.TOY_HD128, 333
    wl = inputs.Workload("host", shape, 1, seq, 200, 90, "random", 16, 0.2, seed=6)
    w, status = inputs.make_weights(shape, seed=6, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    mask = inputs.make_mask(wl)
    h0 = inputs.make_h0(w["embed"].cpu(), inputs.make_tokens(wl, mask))
    torch.empty(1 << 28, dtype=torch.uint8, device="cuda")          # torch keeps this for the workspace
    older()
    ctx = binding.Context(binding.make_config(shape, 1, seq), w)
    h0, mask = h0.contiguous().pin_memory(), mask.contiguous().pin_memory()
    hid, off = torch.zeros(seq, shape.d_model, dtype=torch.bfloat16).pin_memory(), torch.zeros(2, dtype=torch.int32).pin_memory()
    ctx.step_host(h0, mask, seq, 1.0)
    for _ in range(4):                                              # buffers in place once few rows are expected
        older()
        ctx.step_host(h0, mask, 16, 0.1, hidden_out=hid, row_off=off)
    older()
    binding.d2c_op_wait_probe(status, limit_cycles=1000)
    with contextlib.suppress(RuntimeError):                         # (torch reports the older error once and forgets it)
        torch.zeros(1, device="cuda").add_(1)
    assert status.tolist()[:2] == [binding.D2C_ETIMEOUT, 99]


@pytest.mark.parametrize("flags", [0, 1, 4])
def test_logits_that_are_not_numbers_reach_the_confidences(flags):
    """One row of the LM head that is not a number: every confidence is not a number, and the tokens are the best of the
    others.  A hidden state that is not a number: no logit has a maximum, and no token is made up from the padding."""
    shape, seq = replace(inputs.TOY_HD128, vocab=1002), 200          # the last 128 features are not all there
    wl = inputs.Workload("nan", shape, 1, seq, 100, 60, "random", 16, 0.2, seed=6)
    w = inputs.make_weights(shape, seed=6, device="cuda")
    mask = inputs.make_mask(wl)
    h0, mask = inputs.make_h0(w["embed"].cpu(), inputs.make_tokens(wl, mask)).cuda(), mask.cuda()
    at = mask[0].nonzero().flatten()
    def run(w, h0):
        ctx = binding.Context(binding.make_config(shape, 1, seq, flags=flags), w)
        ctx.step(h0, mask, seq, 1.0)
        ctx.sync_status()
        return ctx.view("conf", 1, seq)[0][at].clone(), ctx.view("pred", 1, seq)[0][at].clone()
    conf, pred = run(w, h0)
    assert bool(torch.isfinite(conf).all())
    bad = dict(w, w_lm=w["w_lm"].clone())
    unused = next(t for t in range(200, 300) if not bool((pred == t).any()))
    bad["w_lm"][unused] = float("nan")
    conf2, pred2 = run(bad, h0)
    assert bool(torch.isnan(conf2).all()) and torch.equal(pred, pred2)
    nan_h0 = h0.clone()
    nan_h0[:] = float("nan")
    conf3, pred3 = run(w, nan_h0)
    assert bool(torch.isnan(conf3).all()) and bool((pred3 == 0x7fffffff).all())


@pytest.mark.parametrize("vocab", [1024, 1018, 200])
def test_logits_of_small_steps_that_are_not_numbers_or_infinite(vocab):
    """The same of a small model, in one launch and in separate kernels: a feature that is not a number, hidden states that are not, one
    that is infinite either way.  What is a number and the tokens are the same in each."""
    shape, seq = replace(inputs.TOY, vocab=vocab), 112
    wl = inputs.Workload("nan", shape, 1, seq, 40, 60, "random", 16, 0.2, seed=6)
    w = inputs.make_weights(shape, seed=6, device="cuda")
    mask = inputs.make_mask(wl)
    h0, mask = torch.randn(1, seq, shape.d_model, generator=torch.Generator().manual_seed(3)), mask.cuda()
    h0[0, :, 3] = 30.0 * (1 - 2 * (torch.arange(seq) % 2))           # (far more than a layer adds: the sign stays)
    h0 = h0.to(torch.bfloat16).cuda()
    at = mask[0].nonzero().flatten()
    def run(w, h0, flags):
        ctx = binding.Context(binding.make_config(shape, 1, seq, flags=flags), w)
        ctx.step(h0, mask, seq, 1.0)
        ctx.sync_status()
        return ctx.view("conf", 1, seq)[0][at].clone(), ctx.view("pred", 1, seq)[0][at].clone()
    kinds = (0, 16, 1 | 2)                                           # one launch, separate kernels, portable ones
    good = [run(w, h0, f) for f in kinds]
    unused = next(t for t in range(5, vocab) if not any(bool((pred == t).any()) for _, pred in good))
    bad, inf = (dict(w, w_lm=w["w_lm"].clone()) for _ in range(2))
    bad["w_lm"][unused] = float("nan")
    inf["w_lm"][unused] = 0.0
    inf["w_lm"][unused][3] = float("inf")                            # its logits are +inf or -inf by the sign of one element
    nan_h0 = h0.clone()
    nan_h0[:] = float("nan")
    results = []
    for f, (conf, pred) in zip(kinds, good):
        assert bool(torch.isfinite(conf).all())
        conf2, pred2 = run(bad, h0, f)
        assert bool(torch.isnan(conf2).all()) and torch.equal(pred, pred2), f
        conf3, pred3 = run(w, nan_h0, f)
        assert bool(torch.isnan(conf3).all()) and bool((pred3 == 0x7fffffff).all()), f
        results.append(run(inf, h0, f))
    up = results[0][1] == unused
    assert bool(up.any()) and bool((~up).any())
    for conf, pred in results:
        assert torch.equal(pred == unused, up) and torch.equal(torch.isnan(conf), up)
        torch.testing.assert_close(conf[~up], results[2][0][~up], rtol=3e-2, atol=0)


@pytest.mark.parametrize("rule", [0, 1, 2])
def test_commit_passes_over_rows_that_predict_no_token(rule):
    """One sequence of two has hidden states that are not numbers: nothing of it is committed (its predictions are no rows of
    the embedding table), the other goes on as alone."""
    shape, seq = inputs.TOY_HD128, 200
    wl = inputs.Workload("nan", shape, 2, seq, 100, 60, "random", 16, 0.2, seed=6)
    w = inputs.make_weights(shape, seed=6, device="cuda")
    masks = inputs.make_mask(wl)
    tokens = inputs.make_tokens(wl, masks)
    h0 = inputs.make_h0(w["embed"].cpu(), tokens).cuda()
    out = []
    for bad in (False, True):
        x, mask, tok = h0.clone(), masks.cuda(), tokens.int().cuda()
        if bad:
            x[0] = float("nan")
        ctx = binding.Context(binding.make_config(shape, 2, seq), w)
        ctx.step(x, mask, seq, 1.0)
        committed = torch.full((2,), -5, dtype=torch.int32, device="cuda")
        ctx.commit(w["embed"], x, mask, tok, committed, rule=rule, threshold=0.0)
        ctx.sync_status()
        out.append((committed.tolist(), mask.cpu(), tok.cpu(), x.cpu()))
    (c, m, t, x), (c2, m2, t2, x2) = out
    assert c[0] >= 0 and c2 == [-1, c[1]]
    assert torch.equal(m2[0], masks[0]) and torch.equal(t2[0], tokens[0].int()) and bool(x2[0].isnan().all())
    assert torch.equal(m2[1], m[1]) and torch.equal(t2[1], t[1]) and torch.equal(x2[1], x[1])


def test_a_host_call_that_fails_late_has_let_go_of_its_buffers():
    """The copy of the last result is refused (its buffer is registered in part) when the step is already enqueued: when the
    call comes back with its error, nothing that it enqueued runs any more, and the error is not left for the next caller."""
    shape, batch, seq = inputs.TOY, 3, 8192                          # (results above 64 KB are copied)
    wl = inputs.Workload("late", shape, batch, seq, 8000, 100, "random", 16, 0.1, seed=6)
    w = inputs.make_weights(shape, seed=6, device="cuda")
    mask = inputs.make_mask(wl)
    h0 = inputs.make_h0(w["embed"].cpu(), inputs.make_tokens(wl, mask)).contiguous().pin_memory()
    mask, hid = mask.contiguous().pin_memory(), torch.zeros(batch * seq, shape.d_model, dtype=torch.bfloat16).pin_memory()
    off = torch.zeros(batch + 1, dtype=torch.int32).pin_memory()
    conf = torch.zeros(batch, seq).pin_memory()
    ctx = binding.Context(binding.make_config(shape, batch, seq), w)
    ctx.step_host(h0, mask, seq, 1.0, hidden_out=hid, row_off=off, conf=conf)
    want = hid.clone()
    mem = mmap.mmap(-1, batch * seq * 4)
    base, rt = ctypes.addressof(ctypes.c_char.from_buffer(mem)), torch.cuda.cudart()
    assert int(rt.cudaHostRegister(base, mmap.PAGESIZE, 0)) == 0
    try:
        part = torch.frombuffer(mem, dtype=torch.float32).view(batch, seq)
        hid.zero_()
        with pytest.raises(binding.D2cError) as e:
            ctx.step_host(h0, mask, seq, 1.0, hidden_out=hid, row_off=off, conf=part)
        idle = torch.cuda.current_stream().query()
        assert e.value.code == binding.D2C_ECUDA and idle
        assert torch.equal(hid, want)                                # it had been copied, and will not change any more
        assert int(torch.zeros(4, device="cuda").add_(1).sum()) == 4
        with pytest.raises(binding.D2cError) as e:                   # a bad count is refused before anything is enqueued
            ctx.step_host(h0, mask, 4, 0.1, forced=torch.zeros(1, dtype=torch.int32), forced_off=torch.tensor([0, 0, 0, -1], dtype=torch.int32))
        assert e.value.code == binding.D2C_EINVAL and torch.cuda.current_stream().query()
        hid.zero_()
        ctx.step_host(h0, mask, seq, 1.0, hidden_out=hid, row_off=off, conf=conf)
        assert torch.equal(hid, want)
    finally:
        torch.cuda.synchronize()
        rt.cudaHostUnregister(base)
