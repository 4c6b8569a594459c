"""Parity of the CUDA path (through the C ABI) against the CPU oracle on seeded inputs.

Discrete results (expert ids, permutation, counts, integer reuse scores, resident sets,
counters) must match bit for bit; gate scores are fp32 values computed in the same operation
order and must also match bit for bit; the layer output (bf16 on the GPU, fp64 in the oracle)
must satisfy max-abs error <= 2e-2 and relative L2 error <= 1e-2.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import OracleStack  # noqa: E402
from paper_2609_33385_b200 import synth  # noqa: E402

pytestmark = pytest.mark.gpu

MAX_ABS, REL_L2 = 2e-2, 1e-2


def _runner(w, **kw):
    from paper_2609_33385_b200 import build
    build.build()
    from paper_2609_33385_b200.runner import StackRunner
    return StackRunner(w, **kw)


def _oracle_for(run, caps, policy="priority"):
    w = run.w
    st = OracleStack(w.n_layers, w.hidden, w.n_experts, w.top_k, w.intermediate, caps, policy=policy)
    for l in range(w.n_layers):
        st.register_router(l, run.router_bits[l], run.bias[l])
        if getattr(run, "fp8", False):
            st.register_experts_fp8(l, run.layer_blobs(l))
        else:
            st.register_experts(l, run.layer_blobs(l))
    return st


def _check_out(out_bits, ref, what=""):
    got = synth.bf16_bits_to_f32(out_bits).astype(np.float64)
    err = np.abs(got - ref).max() if ref.size else 0.0
    rel = np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-30) if ref.size else 0.0
    assert err <= MAX_ABS and rel <= REL_L2, f"{what}: max-abs {err:.3e}, rel-L2 {rel:.3e}"
    return err, rel


def _check_step(run, layer, n_tokens, out_t, ref, check_out=True):
    from paper_2609_33385_b200.runner import dev_to_bits
    dbg = run.ctx.debug_last(layer, n_tokens)
    e = run.w.n_experts
    assert np.array_equal(dbg["ids"], ref["ids"]), "expert ids differ"
    assert np.array_equal(dbg["gate"].view(np.uint32), ref["gate"].view(np.uint32)), "gate scores differ"
    assert np.array_equal(dbg["counts"], ref["counts"])
    assert np.array_equal(dbg["perm"], ref["perm"]), "permutation differs"
    assert [int(v) for v in dbg["scores"]] == list(ref["scores"]), "reuse scores differ"
    assert set(np.flatnonzero(dbg["resident_before"])) == ref["resident_before"]
    assert set(np.flatnonzero(dbg["resident_after"])) == ref["resident_after"]
    dbp = run.ctx.debug_perm(layer, n_tokens)
    assert np.array_equal(dbp["offsets"], ref["offsets"]), "offsets differ"
    assert np.array_equal(dbp["pos"], ref["pos"]), "inverse permutation differs"
    if n_tokens:
        logits = run.ctx.debug_logits(layer, n_tokens)
        assert np.array_equal(logits.view(np.uint32), ref["logits"].view(np.uint32)), "logits differ"
    if check_out:
        _check_out(dev_to_bits(out_t), ref["out"], f"layer {layer}")
    assert len(dbg["counts"]) == e


def _check_stats(run, ora):
    for l in range(run.w.n_layers):
        a, b = run.ctx.stats(l), ora.stats(l)
        assert (a.steps, a.hits, a.misses, a.bytes_moved, a.evictions, a.active_experts, a.assignments,
                a.fills_reused, a.ideal_hits) == \
               (b.steps, b.hits, b.misses, b.bytes_moved, b.evictions, b.active_experts, b.assignments,
                b.fills_reused, b.ideal_hits)
    a, b = run.ctx.stats(-1), ora.stats(-1)
    assert (a.hits, a.misses, a.bytes_moved) == (b.hits, b.misses, b.bytes_moved)


def _run_stack(run, ora, check_out=True):
    """Replay mode: the oracle is fed the bf16 inputs the GPU saw at every call."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = run.w
    dev = run.device
    out = torch.empty((w.tokens, w.hidden), dtype=torch.bfloat16, device=dev)
    bufs = [torch.empty_like(out), torch.empty_like(out)]
    for b, i, h_bits, conf in synth.denoise_inputs(w):
        x = bits_to_dev(h_bits, dev)
        c = torch.from_numpy(conf).to(dev)
        for l in range(w.n_layers):
            run.step(l, x, c, out)
            ref = ora.denoise_step(l, dev_to_bits(x), conf)
            _check_step(run, l, w.tokens, out, ref, check_out)
            nxt = bufs[l & 1]
            run.ctx.residual_add(x.data_ptr(), out.data_ptr(), nxt.data_ptr(), x.numel())
            # the residual kernel: bf16(x + out) with one rounding
            exp = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(dev_to_bits(x)) +
                                         synth.bf16_bits_to_f32(dev_to_bits(out)))
            assert np.array_equal(dev_to_bits(nxt), exp)
            x = nxt
    _check_stats(run, ora)


@pytest.mark.parametrize("ffn_impl", [1, 0], ids=["ffn-plain", "ffn-tcgen05"])
def test_tiny_stack_elementwise(ffn_impl):
    w = synth.tiny()
    run = _runner(w, capacity=[3, 5], ffn_impl=ffn_impl)
    try:
        _run_stack(run, _oracle_for(run, [3, 5]))
    finally:
        run.close()


@pytest.mark.parametrize("ffn_impl", [1, 0], ids=["ffn-plain", "ffn-tcgen05"])
def test_config1_full_run(ffn_impl):
    w = synth.config(0)                        # hidden 512, 16 experts top-2, I 1024, 32 tokens
    run = _runner(w, ffn_impl=ffn_impl)
    try:
        _run_stack(run, _oracle_for(run, [w.capacity]))
        st = run.ctx.stats()
        assert st.steps == w.iters and st.misses > 0 and st.hits > 0
    finally:
        run.close()


@pytest.mark.parametrize("n_tokens", [0, 1, 7, 33, 150])
def test_ragged_token_counts(n_tokens):
    """Token counts that leave experts empty, span several 16-row tiles and end in a ragged tail."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=6, top_k=3, hidden=512, intermediate=256)
    run = _runner(w, capacity=[2], max_tokens=160)
    ora = _oracle_for(run, [2])
    try:
        for rep in range(2):
            h_bits, conf = synth.flat_tokens(w, n_tokens, rep)
            x = bits_to_dev(h_bits, run.device) if n_tokens else torch.empty((0, w.hidden), dtype=torch.bfloat16, device=run.device)
            c = torch.from_numpy(conf).to(run.device)
            out = torch.zeros((max(n_tokens, 1), w.hidden), dtype=torch.bfloat16, device=run.device)[:n_tokens]
            run.step(0, x, c, out)
            ref = ora.denoise_step(0, h_bits.reshape(n_tokens, w.hidden), conf)
            _check_step(run, 0, n_tokens, out, ref)
        _check_stats(run, ora)
    finally:
        run.close()


@pytest.mark.parametrize("n_experts,n_tokens", [(64, 5), (64, 200), (64, 310), (128, 33), (128, 256), (128, 300)])
def test_gate_with_64_and_128_experts(n_experts, n_tokens):
    """The expert counts of the benchmark configurations at a small hidden size, with one, two and four
    tokens per CTA of the few-token gate kernel (several passes over the experts per warp): logits,
    ids, gate scores bit for bit; and the two layers as one iteration, whose second gate kernel
    carries the first layer's combine."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=2, n_experts=n_experts, top_k=8, hidden=768, intermediate=128)
    run = _runner(w, capacity=[n_experts // 2, n_experts // 2], max_tokens=n_tokens)
    ora = _oracle_for(run, [n_experts // 2, n_experts // 2])
    try:
        h_bits, conf = synth.flat_tokens(w, n_tokens, 3)
        c = torch.from_numpy(conf).to(run.device)
        x = bits_to_dev(h_bits, run.device)
        for layer in range(2):
            out = torch.empty((n_tokens, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(layer, x, c, out)
            ref = ora.denoise_step(layer, dev_to_bits(x), conf)
            _check_step(run, layer, n_tokens, out, ref)
            nxt = torch.empty_like(out)
            run.ctx.residual_add(x.data_ptr(), out.data_ptr(), nxt.data_ptr(), x.numel())
            x = nxt
        # the same two layers as one iteration (the second gate kernel carries the first layer's combine)
        run2 = _runner(w, capacity=[n_experts // 2, n_experts // 2], max_tokens=n_tokens)
        try:
            y = torch.empty((n_tokens, w.hidden), dtype=torch.bfloat16, device=run.device)
            x0 = bits_to_dev(h_bits, run.device)
            run2.ctx.denoise_iteration(x0.data_ptr(), c.data_ptr(), n_tokens, y.data_ptr())
            assert np.array_equal(dev_to_bits(y), dev_to_bits(x))
        finally:
            run2.close()
    finally:
        run.close()


@pytest.mark.parametrize("n", [700, 2100])
def test_many_tokens_per_expert_multi_tile(n):
    """More than 256 rows for one expert: several N tiles per expert in both FFN kernels; the
    larger case also takes the many-token variants of the gate and gather kernels."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=256, intermediate=128)
    run = _runner(w, capacity=[4], max_tokens=n)
    ora = _oracle_for(run, [4])
    try:
        h_bits, conf = synth.flat_tokens(w, n, 7)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)
        ref = ora.denoise_step(0, h_bits, conf)
        assert ref["counts"].max() > 256
        _check_step(run, 0, n, out, ref)
    finally:
        run.close()


def _rows_copied_by_the_permutation(run, n):
    """Did the permutation kernel of the steps since the last reading copy the token rows (by its bytes in the profile)?"""
    p = run.ctx.profile_read()["permute"]
    assert p["launches"] > 0
    return p["bytes"] > p["launches"] * n * run.w.top_k * 12


@pytest.mark.parametrize("n", [700, 2100])
def test_cta_pair_ffn_form_many_tokens(n):
    """Token tiles of 256 rows with hidden a multiple of 512 and intermediate a multiple of 256: the
    expert FFN runs on CTA pairs (cta_group::2), each CTA holding half of a token tile.  Ragged
    last tiles, several tiles per expert; against the oracle, against the one-CTA form
    (OLED_OPT_FFN_PAIRS 0), which accumulates every output in the same order, and the one-launch
    pair form (gate/up items, then down items behind per-expert counters) against the two-launch
    one (OLED_OPT_FUSE_FFN 0)."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=512, intermediate=256)
    run = _runner(w, capacity=[4], max_tokens=n)
    ora = _oracle_for(run, [4])
    try:
        h_bits, conf = synth.flat_tokens(w, n, 9)
        c = torch.from_numpy(conf).to(run.device)
        ref = ora.denoise_step(0, h_bits, conf)
        assert ref["counts"].max() > 256
        outs = []
        for pairs, fuse in ((1, 1), (0, 1), (1, 0)):   # one launch on pairs; one CTA per tile; two launches on pairs
            run.ctx.set_option(binding.OPT_FFN_PAIRS, pairs)
            run.ctx.set_option(binding.OPT_FUSE_FFN, fuse)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, bits_to_dev(h_bits, run.device), c, out)
            _check_step(run, 0, n, out, ref)
            outs.append(out.float().cpu().numpy().astype(np.float64))
            run.ctx.reset_cache()
        assert np.linalg.norm(outs[0] - outs[1]) <= 1e-3 * np.linalg.norm(outs[1])
        assert np.array_equal(outs[0], outs[2])   # the same items in the same arithmetic, one launch or two
        # token rows gathered by the FFN launch itself (forced: the matrices are small; a many-token step, n = 2100)
        # or by the permutation kernel in front: the same operands
        run.ctx.set_option(binding.OPT_PROFILE, 1)
        for fuse in (1, 0):
            for gather in (2, 0):
                run.ctx.set_option(binding.OPT_FFN_PAIRS, 1)
                run.ctx.set_option(binding.OPT_FUSE_FFN, fuse)
                run.ctx.set_option(binding.OPT_GATHER_IN_FFN, gather)
                run.step(0, bits_to_dev(h_bits, run.device), c, out)   # (cold: the experts are fetched)
                _check_step(run, 0, n, out, ref)
                run.ctx.profile_read()
                out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
                run.step(0, bits_to_dev(h_bits, run.device), c, out)
                if n == 2100:
                    assert _rows_copied_by_the_permutation(run, n) == (gather == 0)
                assert np.array_equal(outs[0], out.float().cpu().numpy().astype(np.float64))
                run.ctx.reset_cache()
    finally:
        run.close()


@pytest.mark.parametrize("hidden", [512, 4608])
def test_gather_in_ffn_with_cache_misses(hidden):
    """A many-token step with misses whose FFN launches gather their own token rows (forced: the matrices are small): those
    over the fetched experts as well (token tile 256 whatever their counts), ragged tiles included.  hidden 4608: a
    row is moved as two pieces (8192 + 1024 bytes)."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    n = 2100
    # (weights scaled with the contraction length, so that the outputs stay of order one)
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=hidden, intermediate=256,
                   weight_std=0.05 * (512 / hidden) ** 0.5)
    run = _runner(w, capacity=[2], max_tokens=n)
    ora = _oracle_for(run, [2])
    try:
        run.ctx.set_option(binding.OPT_GATHER_IN_FFN, 2)
        run.ctx.set_option(binding.OPT_PROFILE, 1)
        got = []
        for seed in (9, 10):
            h_bits, conf = synth.flat_tokens(w, n, seed)
            ref = ora.denoise_step(0, h_bits, conf)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device), out)
            _check_step(run, 0, n, out, ref)
            got.append(dev_to_bits(out).copy())
        assert run.ctx.stats().misses > 0
        assert not _rows_copied_by_the_permutation(run, n)
        # the same two steps with the rows copied by the permutation kernel: the same bits
        run.ctx.reset_cache()
        run.ctx.set_option(binding.OPT_GATHER_IN_FFN, 0)
        for i, seed in enumerate((9, 10)):
            h_bits, conf = synth.flat_tokens(w, n, seed)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device), out)
            assert np.array_equal(got[i], dev_to_bits(out))
        assert _rows_copied_by_the_permutation(run, n)
    finally:
        run.close()


def test_output_bit_identical_at_every_capacity():
    """Offloading is lossless (Sec. 5.1): routing and output do not depend on the capacity."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1, blocks=1, iters=4, n_experts=8, top_k=2)
    outs, miss = [], []
    for cap in (1, 3, 8):
        run = _runner(w, capacity=[cap])
        try:
            res = []
            for _, _, h_bits, conf in synth.denoise_inputs(w):
                x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
                out = torch.empty((w.tokens, w.hidden), dtype=torch.bfloat16, device=run.device)
                run.step(0, x, c, out)
                res.append((dev_to_bits(out).copy(), run.ctx.debug_last(0, w.tokens)["ids"].copy()))
            outs.append(res)
            miss.append(run.ctx.stats().misses)
        finally:
            run.close()
    for res in outs[1:]:
        for (o0, i0), (o1, i1) in zip(outs[0], res):
            assert np.array_equal(i0, i1) and np.array_equal(o0, o1)
    assert miss[0] >= miss[1] >= miss[2]


def test_iteration_entry_points_match_layer_by_layer_steps():
    """oled_denoise_iteration (device and host buffers) == steps + residual adds, bit for bit."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=3, n_experts=8, top_k=2)
    runs = [_runner(w, capacity=[3, 4, 2]) for _ in range(3)]
    try:
        dev = runs[0].device
        out = torch.empty((w.tokens, w.hidden), dtype=torch.bfloat16, device=dev)
        bufs = [torch.empty_like(out), torch.empty_like(out)]
        for _, _, h_bits, conf in synth.denoise_inputs(w):
            x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
            ref = dev_to_bits(runs[0].iteration(x, c, bufs, out)).copy()
            y = torch.empty_like(out)
            runs[1].ctx.denoise_iteration(x.data_ptr(), c.data_ptr(), w.tokens, y.data_ptr())
            assert np.array_equal(dev_to_bits(y), ref)
            hx = torch.from_numpy(h_bits.view(np.int16)).pin_memory()
            hc = torch.from_numpy(conf).pin_memory()
            hy = torch.empty((w.tokens, w.hidden), dtype=torch.int16).pin_memory()
            runs[2].ctx.denoise_iteration_host(hx.data_ptr(), hc.data_ptr(), w.tokens, hy.data_ptr())
            assert np.array_equal(hy.numpy().view(np.uint16), ref)
        assert runs[0].ctx.stats() == runs[1].ctx.stats() == runs[2].ctx.stats()
        assert runs[0].ctx.stats().steps == 3 * w.iters * w.blocks
    finally:
        for r in runs:
            r.close()


def test_l2_prefetch_across_layers_changes_no_bit():
    """OLED_OPT_L2_PREFETCH only calls weights into L2: with all experts resident (no miss, so the
    prefetch kernel runs behind every layer; value 2 lifts the stream-length condition the tiny
    shape would not meet) the iterations' outputs and statistics equal those with it off."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=3, n_experts=8, top_k=2)
    runs = [_runner(w, capacity=[8, 8, 8]) for _ in range(2)]
    try:
        runs[0].ctx.set_option(binding.OPT_L2_PREFETCH, 2)
        runs[1].ctx.set_option(binding.OPT_L2_PREFETCH, 0)
        dev = runs[0].device
        for _, _, h_bits, conf in synth.denoise_inputs(w):
            x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
            ys = []
            for r in runs:
                y = torch.empty((w.tokens, w.hidden), dtype=torch.bfloat16, device=dev)
                r.ctx.denoise_iteration(x.data_ptr(), c.data_ptr(), w.tokens, y.data_ptr())
                ys.append(dev_to_bits(y).copy())
            assert np.array_equal(ys[0], ys[1])
        assert runs[0].ctx.stats() == runs[1].ctx.stats()
        assert runs[0].ctx.launch_count() > runs[1].ctx.launch_count()   # the prefetch kernel did run
    finally:
        for r in runs:
            r.close()


def test_host_buffer_entry_point_matches_device_entry_point():
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1)
    run_d, run_h = _runner(w, capacity=[3]), _runner(w, capacity=[3])
    try:
        for _, _, h_bits, conf in synth.denoise_inputs(w):
            x, c = bits_to_dev(h_bits, run_d.device), torch.from_numpy(conf).to(run_d.device)
            out = torch.empty((w.tokens, w.hidden), dtype=torch.bfloat16, device=run_d.device)
            run_d.step(0, x, c, out)
            hx = torch.from_numpy(h_bits.view(np.int16)).pin_memory()
            hc = torch.from_numpy(conf).pin_memory()
            ho = torch.empty((w.tokens, w.hidden), dtype=torch.int16).pin_memory()
            run_h.step_host(0, hx, hc, ho)
            assert np.array_equal(ho.numpy().view(np.uint16), dev_to_bits(out))
        assert run_d.ctx.stats() == run_h.ctx.stats()
    finally:
        run_d.close()
        run_h.close()


def test_errors_are_codes_not_crashes():
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1)
    ctx = binding.OledContext(1, w.hidden, w.n_experts, w.top_k, w.intermediate, 8, [2])
    try:
        x = torch.zeros((8, w.hidden), dtype=torch.bfloat16, device="cuda:0")
        c = torch.zeros(8, device="cuda:0")
        out = torch.zeros_like(x)
        assert ctx.denoise_step_rc(0, x.data_ptr(), c.data_ptr(), 8, out.data_ptr()) == binding.ERR_NOT_REGISTERED
        wr, _ = synth.router_weights(w, 0)
        wr_d = bits_to_dev(wr, "cuda:0")
        ctx.register_router(0, wr_d.data_ptr())
        pageable = torch.zeros((w.n_experts, w.expert_elems), dtype=torch.int16)
        with pytest.raises(binding.OledError) as ei:
            ctx.register_experts(0, pageable.data_ptr(), w.expert_bytes)
        assert ei.value.code == binding.ERR_NOT_PINNED
        pinned = torch.zeros((w.n_experts, w.expert_elems), dtype=torch.int16).pin_memory()
        with pytest.raises(binding.OledError) as ei:
            ctx.register_experts(0, pinned.data_ptr(), w.expert_bytes - 16)
        assert ei.value.code == binding.ERR_INVALID_ARG
        ctx.register_experts(0, pinned.data_ptr(), w.expert_bytes)
        assert ctx.denoise_step_rc(0, x.data_ptr(), c.data_ptr(), 9, out.data_ptr()) == binding.ERR_TOO_MANY_TOKENS
        assert ctx.denoise_step_rc(1, x.data_ptr(), c.data_ptr(), 8, out.data_ptr()) == binding.ERR_INVALID_ARG
        assert ctx.denoise_step_rc(0, x.data_ptr(), c.data_ptr(), 8, x.data_ptr()) == binding.ERR_INVALID_ARG
        assert ctx.denoise_step_rc(0, None, c.data_ptr(), 8, out.data_ptr()) == binding.ERR_INVALID_ARG
        # rows are moved with 16-byte vector accesses: a view that starts inside one is refused
        big = torch.zeros(8 * w.hidden + 8, dtype=torch.bfloat16, device="cuda:0")
        assert ctx.denoise_step_rc(0, big[4:].data_ptr(), c.data_ptr(), 8, out.data_ptr()) == binding.ERR_INVALID_ARG
        assert ctx.denoise_step_rc(0, x.data_ptr(), c.data_ptr(), 8, big[4:].data_ptr()) == binding.ERR_INVALID_ARG
        assert ctx.denoise_step_rc(0, x.data_ptr(), c.data_ptr(), 8, out.data_ptr()) == binding.OLED_OK
        ctx.synchronize()
        assert float(out.float().abs().max()) == 0.0          # zero weights -> zero output
        with pytest.raises(binding.OledError):
            binding.OledContext(1, 250, 8, 2, 128, 8, [2])     # hidden not a multiple of 256
        with pytest.raises(binding.OledError):
            binding.OledContext(1, 256, 8, 2, 128, 8, [9])     # capacity > E
    finally:
        ctx.destroy()


def test_reset_cache_returns_to_cold_state():
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1)
    run = _runner(w, capacity=[w.n_experts])
    try:
        h_bits, conf = synth.flat_tokens(w, 5)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((5, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)
        m1 = run.ctx.stats().misses
        run.step(0, x, c, out)
        assert run.ctx.stats().misses == m1 and m1 > 0        # second identical step: all hits
        run.ctx.reset_cache()
        assert run.ctx.stats().steps == 0
        run.step(0, x, c, out)
        assert run.ctx.stats().misses == m1
    finally:
        run.close()


@pytest.mark.parametrize("policy", ["lru", "lfu"])
def test_comparison_policies_match_oracle(policy):
    """LRU / LFU retention through the real step: resident sets, counters and outputs."""
    w = synth.tiny(n_layers=2, blocks=2, iters=4, n_experts=8, top_k=2)
    run = _runner(w, capacity=[3, 2], policy=policy)
    try:
        _run_stack(run, _oracle_for(run, [3, 2], policy=policy))
    finally:
        run.close()


def test_layer_adaptive_sizing_through_the_iteration_entry_point():
    """oled_denoise_iteration with a refresh period of 2: capacities, resident sets and counters
    follow the oracle's layer-adaptive sizing; outputs stay within tolerance."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=3, blocks=3, iters=3, n_experts=8, top_k=2)
    caps = [3, 3, 3]
    run = _runner(w, capacity=caps, adapt_period=2, staging_slots=8)
    ora = _oracle_for(run, caps)
    try:
        dev = run.device
        y = torch.empty((w.tokens, w.hidden), dtype=torch.bfloat16, device=dev)
        out = torch.empty_like(y)
        bufs = [torch.empty_like(y), torch.empty_like(y)]
        shadow = _runner(w, capacity=caps, staging_slots=8)       # same inputs, step by step, for replay
        changed = False
        for it, (_, _, h_bits, conf) in enumerate(synth.denoise_inputs(w)):
            x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
            run.ctx.denoise_iteration(x.data_ptr(), c.data_ptr(), w.tokens, y.data_ptr())
            # replay the same iteration layer by layer on the shadow context to feed the oracle
            xs = x
            for l in range(w.n_layers):
                shadow.step(l, xs, c, out)
                ora.denoise_step(l, dev_to_bits(xs), conf)
                nxt = bufs[l & 1]
                shadow.ctx.residual_add(xs.data_ptr(), out.data_ptr(), nxt.data_ptr(), xs.numel())
                xs = nxt
            assert np.array_equal(dev_to_bits(y), dev_to_bits(xs))   # capacity never changes outputs
            if (it + 1) % 2 == 0:
                want = ora.adapt_capacity()
                assert run.ctx.get_capacity() == want and sum(want) == sum(caps)
                changed = changed or want != caps
            for l in range(w.n_layers):
                a, b = run.ctx.stats(l), ora.stats(l)
                assert (a.hits, a.misses, a.evictions, a.fills_reused) == \
                       (b.hits, b.misses, b.evictions, b.fills_reused), (it, l)
        assert changed, "the allocation never moved: the test exercises nothing"
        shadow.close()
    finally:
        run.close()


def test_bounded_device_wait_reports_timeout_and_context_survives():
    """Failure path without a fault: the FFN kernels' load producers are told to issue nothing, so
    the consumers' bounded waits run out; the kernels flag it and return, the host reads
    OLED_ERR_TIMEOUT, and after oled_clear_status() the same context computes correct results."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1)
    run = _runner(w, capacity=[w.n_experts])
    ora = _oracle_for(run, [w.n_experts])
    try:
        h_bits, conf = synth.flat_tokens(w, 5)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((5, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)                                   # warm: everything resident
        ref = ora.denoise_step(0, h_bits, conf)
        run.ctx.synchronize()
        run.ctx.set_option(binding.OPT_TEST_WITHHOLD_LOADS, 1)
        run.step(0, x, c, out)                                   # hits only: one FFN launch pair
        assert run.ctx.synchronize_rc() == binding.ERR_TIMEOUT
        assert run.ctx.synchronize_rc() == binding.ERR_TIMEOUT   # sticky until cleared
        run.ctx.set_option(binding.OPT_TEST_WITHHOLD_LOADS, 0)
        run.ctx.clear_status()
        assert run.ctx.synchronize_rc() == binding.OLED_OK
        ora.denoise_step(0, h_bits, conf)                        # keep the oracle's counters in step
        run.step(0, x, c, out)
        _check_out(dev_to_bits(out), ora.denoise_step(0, h_bits, conf)["out"])
        ns, runs = run.ctx.policy_time()
        assert runs == 3 and ns > 0
    finally:
        run.close()


def test_bounded_device_wait_in_the_cta_pair_kernel():
    """The same failure path in the many-token FFN on CTA pairs: no item is ever published, the
    bounded waits of every role of both CTAs run out, the cluster's kernels return, the host
    reads OLED_ERR_TIMEOUT, and afterwards the same context is in parity again."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=512, intermediate=256)
    n = 700
    run = _runner(w, capacity=[4], max_tokens=n)
    ora = _oracle_for(run, [4])
    try:
        h_bits, conf = synth.flat_tokens(w, n, 11)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)                                   # warm: everything resident
        ref = ora.denoise_step(0, h_bits, conf)
        assert ref["counts"].max() > 256                         # token tiles of 256 rows: the pair kernel
        _check_out(dev_to_bits(out), ref["out"])
        run.ctx.set_option(binding.OPT_TEST_WITHHOLD_LOADS, 1)
        run.step(0, x, c, out)
        assert run.ctx.synchronize_rc() == binding.ERR_TIMEOUT
        run.ctx.set_option(binding.OPT_TEST_WITHHOLD_LOADS, 0)
        run.ctx.clear_status()
        assert run.ctx.synchronize_rc() == binding.OLED_OK
        ora.denoise_step(0, h_bits, conf)                        # keep the oracle's counters in step
        run.step(0, x, c, out)
        _check_out(dev_to_bits(out), ora.denoise_step(0, h_bits, conf)["out"])
    finally:
        run.close()


def test_self_check_is_silent_on_valid_steps_and_flags_a_corrupted_permutation():
    """OLED_OPT_SELF_CHECK: the checking kernels find nothing on valid steps (parity unchanged, guard
    words intact); with the first two sorted rows exchanged by the test aid - both still valid
    rows, so nothing faults - the next synchronising call returns OLED_ERR_SELF_CHECK and the
    report names the broken invariant; after oled_clear_status() the context is in parity again."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(blocks=1, iters=3)
    run = _runner(w, capacity=[3, 5], max_tokens=max(w.tokens, 9))
    ora = _oracle_for(run, [3, 5])
    try:
        run.ctx.set_option(binding.OPT_SELF_CHECK, 1)
        _run_stack(run, ora)                                     # every step checked, all in parity
        run.ctx.synchronize()
        assert run.ctx.self_check_report() == ([], -1, 0)
        h_bits, conf = synth.flat_tokens(w, 9, 3)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((9, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.ctx.set_option(binding.OPT_TEST_CORRUPT_PERM, 1)
        run.step(0, x, c, out)
        ora.denoise_step(0, h_bits, conf)                        # keep the oracle's cache state in step
        assert run.ctx.synchronize_rc() == binding.ERR_SELF_CHECK
        names, index, guard = run.ctx.self_check_report()
        assert "inverse" in names and index in (0, 1) and guard == 0
        assert run.ctx.synchronize_rc() == binding.ERR_SELF_CHECK   # sticky until cleared
        run.ctx.set_option(binding.OPT_TEST_CORRUPT_PERM, 0)
        run.ctx.clear_status()
        assert run.ctx.synchronize_rc() == binding.OLED_OK
        run.step(0, x, c, out)
        _check_step(run, 0, 9, out, ora.denoise_step(0, h_bits, conf))
        assert run.ctx.self_check_report() == ([], -1, 0)
    finally:
        run.close()


def test_maximum_expert_count_and_top_k():
    """512 experts (OLED_MAX_EXPERTS) with top-32 (OLED_MAX_TOPK): the widest gate the ABI allows."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=512, top_k=32, hidden=256, intermediate=128)
    run = _runner(w, capacity=[40], max_tokens=8)
    ora = _oracle_for(run, [40])
    try:
        for rep, n in enumerate((3, 8)):
            h_bits, conf = synth.flat_tokens(w, n, 20 + rep)
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, x, c, out)
            _check_step(run, 0, n, out, ora.denoise_step(0, h_bits, conf))
        _check_stats(run, ora)
    finally:
        run.close()


def test_degenerate_routing_cases():
    """Identical tokens (one expert set takes every token), zero confidences (all reuse scores
    zero: retention falls back to the id order) and top-k equal to the number of experts."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=4, top_k=4, hidden=256, intermediate=128)
    run = _runner(w, capacity=[2], max_tokens=40)
    ora = _oracle_for(run, [2])
    try:
        h_bits, conf = synth.flat_tokens(w, 40, 30)
        same = np.repeat(h_bits[:1], 40, axis=0)                       # every token identical
        zero_c = np.zeros(40, np.float32)
        for hb, cf in ((same, conf), (h_bits, zero_c), (same, zero_c)):
            x, c = bits_to_dev(hb, run.device), torch.from_numpy(cf).to(run.device)
            out = torch.empty((40, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, x, c, out)
            ref = ora.denoise_step(0, hb, cf)
            _check_step(run, 0, 40, out, ref)
            assert ref["counts"].tolist() == [40, 40, 40, 40]           # k = E: every expert, every token
        _check_stats(run, ora)
    finally:
        run.close()
    # a single expert set for all tokens with k < E: two experts hold all 2*T assignments
    w2 = synth.tiny(n_layers=1, n_experts=8, top_k=2, hidden=256, intermediate=128)
    run = _runner(w2, capacity=[3], max_tokens=300)
    ora = _oracle_for(run, [3])
    try:
        h_bits, conf = synth.flat_tokens(w2, 300, 31)
        same = np.repeat(h_bits[:1], 300, axis=0)
        x, c = bits_to_dev(same, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((300, w2.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)
        ref = ora.denoise_step(0, same, conf)
        assert sorted(ref["counts"].tolist())[-2:] == [300, 300] and ref["counts"].sum() == 600
        _check_step(run, 0, 300, out, ref)
    finally:
        run.close()


def test_non_finite_activations_keep_routing_defined_and_the_context_usable():
    """NaN and Inf in the hidden states: a NaN logit ranks as -inf, so the k ids of every token
    stay distinct and all discrete results still match the oracle; rows of clean tokens are
    unaffected; the next clean step is in full parity."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1)
    run = _runner(w, capacity=[3], max_tokens=40)
    ora = _oracle_for(run, [3])
    try:
        h_bits, conf = synth.flat_tokens(w, 40, 77)
        bad = h_bits.copy()
        bad[3, :] = 0x7FC0      # a whole NaN row
        bad[5, 17] = 0x7FC0     # one NaN element
        bad[7, 1] = 0x7F80      # +Inf
        bad[9, 2] = 0xFF80      # -Inf
        x, c = bits_to_dev(bad, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((40, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)
        with np.errstate(all="ignore"):
            ref = ora.denoise_step(0, bad, conf)
        dbg = run.ctx.debug_last(0, 40)
        assert np.array_equal(dbg["ids"], ref["ids"])
        assert all(len(set(row)) == w.top_k for row in dbg["ids"].tolist())
        assert np.array_equal(np.isnan(dbg["gate"]), np.isnan(ref["gate"]))
        ok = ~np.isnan(ref["gate"])
        assert np.array_equal(dbg["gate"][ok].view(np.uint32), ref["gate"][ok].view(np.uint32))
        assert np.array_equal(dbg["counts"], ref["counts"]) and np.array_equal(dbg["perm"], ref["perm"])
        assert [int(v) for v in dbg["scores"]] == list(ref["scores"])
        assert set(np.flatnonzero(dbg["resident_after"])) == ref["resident_after"]
        clean = [t for t in range(40) if t not in (3, 5, 7, 9)]
        _check_out(dev_to_bits(out)[clean], ref["out"][clean], "clean rows")
        x2 = bits_to_dev(h_bits, run.device)
        run.step(0, x2, c, out)
        _check_step(run, 0, 40, out, ora.denoise_step(0, h_bits, conf))
        _check_stats(run, ora)
    finally:
        run.close()


def test_fp8_expert_store_tiny_stack():
    """fp8 (e4m3 + row scales) expert blobs: same discrete results, outputs within the same
    tolerance of the oracle evaluated on the dequantised weights, half the bytes moved."""
    w = synth.tiny(blocks=2, iters=3)
    run = _runner(w, capacity=[3, 5], fp8=True)
    try:
        ora = _oracle_for(run, [3, 5])
        _run_stack(run, ora)
        st = run.ctx.stats()
        assert st.bytes_moved == st.misses * synth.fp8_blob_bytes(w)
        assert synth.fp8_blob_bytes(w) < 0.55 * w.expert_bytes
    finally:
        run.close()


@pytest.mark.parametrize("direct", [1, 0], ids=["direct", "widening"])
@pytest.mark.parametrize("n", [24, 40, 300, 700, 2100])
def test_fp8_expert_store_token_tile_variants(n, direct):
    """fp8 blobs through every FFN tile form that exists for them (OLED_OPT_FP8_DIRECT): codes read directly, token tiles
    of 32, 48 and 128 rows; codes widened, stacked (token tiles up to 32 rows) and two accumulators (64 and 128
    rows).  700 tokens: several tiles per expert; 2100: more than 4096 assignments, where matrices this small are
    widened in both settings."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=512, intermediate=256)
    run = _runner(w, capacity=[4], max_tokens=n, fp8=True)
    ora = _oracle_for(run, [4])
    try:
        run.ctx.set_option(binding.OPT_FP8_DIRECT, direct)
        h_bits, conf = synth.flat_tokens(w, n, 50)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)
        _check_step(run, 0, n, out, ora.denoise_step(0, h_bits, conf))
    finally:
        run.close()


def test_fp8_direct_form_agrees_with_widening_form_on_wide_range_rows():
    """The form whose MMAs read the e4m3 codes directly, the token rows entering as two e4m3 terms
    after a per-row power-of-two scale, on a block of 24 tokens.  Rows with a wide
    dynamic range (elements 2^-12 below the row's maximum), an all-zero row and a row 2^10 larger
    than the rest: same discrete results, outputs within tolerance of the oracle, and the two
    forms (OLED_OPT_FP8_DIRECT 1 / 0) agree far more closely than either has to with the oracle."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=512, intermediate=256)
    n = 24
    run = _runner(w, capacity=[4], max_tokens=n, fp8=True)
    ora = _oracle_for(run, [4])
    try:
        h_bits, conf = synth.flat_tokens(w, n, 51)
        f = (h_bits.astype(np.uint32) << 16).view(np.float32).copy()
        f[:, ::3] *= 2.0 ** -12          # a third of every row far below the row's maximum
        f[3, :] = 0.0                    # an all-zero row
        f[5, :] *= 2.0 ** 10             # one row far above the others
        h_bits = (f.view(np.uint32) >> 16).astype(np.uint16)   # (scaling by powers of two is exact in bf16)
        c = torch.from_numpy(conf).to(run.device)
        with np.errstate(over="ignore"):   # exp(-a) of the large row's gate values overflows to inf: silu -> -0
            ref = ora.denoise_step(0, h_bits, conf)
        outs = []
        for direct in (1, 0):
            run.ctx.set_option(binding.OPT_FP8_DIRECT, direct)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, bits_to_dev(h_bits, run.device), c, out)
            if direct:
                _check_step(run, 0, n, out, ref, check_out=False)
            outs.append(out.float().cpu().numpy().astype(np.float64))
            run.ctx.reset_cache()
        a, b = outs
        assert np.all(a[3] == 0.0) and np.all(b[3] == 0.0) and np.all(ref["out"][3] == 0.0)
        for t in range(n):   # row by row and relative: the rows differ in scale by orders of magnitude
            den = np.linalg.norm(ref["out"][t])
            if den > 0:
                assert np.linalg.norm(a[t] - ref["out"][t]) / den <= REL_L2, ("direct form against the oracle", t)
                assert np.linalg.norm(b[t] - ref["out"][t]) / den <= REL_L2, ("widening form against the oracle", t)
                assert np.linalg.norm(a[t] - b[t]) / den < 3e-3, ("the two forms", t)
    finally:
        run.close()


@pytest.mark.parametrize("shape,counts,capacity", [((8, 8, 2048, 512), (700, 523), 8), ((8, 8, 2048, 512), (700, 700), 5),
                                                   ((40, 8, 1024, 1024), (530, 1024), 40)])
def test_fp8_codes_read_directly_beyond_4096_assignments(shape, counts, capacity):
    """fp8 steps of more than 4096 assignments with expert matrices of 2^20 elements and more: the segmented permutation
    makes the rows' e4m3 terms, the FFN reads the codes directly over sorted rows and stores bf16 outputs per
    assignment.  Every expert takes several tiles, segments and tiles end raggedly, a row has a wide range of
    magnitudes, one is all zero and one far above the others; capacity 5: fetched experts in launches of their own.
    Parity with the oracle; the same bits when repeated; and no further from the oracle's 64-bit sums than the
    widening form (OLED_OPT_FP8_DIRECT 0), which multiplies the rows as they are.  Both are 2.3e-3 to 2.9e-3 away - bf16
    intermediate rows and outputs, which fall either way in the last place: over 50 shapes and seeds the two errors
    differed by up to 0.03 % from 100 tokens on."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    e, k, h, i = shape
    w = synth.tiny(n_layers=1, n_experts=e, top_k=k, hidden=h, intermediate=i, weight_std=0.02)
    run = _runner(w, capacity=[capacity], max_tokens=max(counts), fp8=True)
    ora = _oracle_for(run, [capacity])
    try:
        assert h * i >= 1 << 20 and min(counts) * k > 4096
        run.ctx.set_option(binding.OPT_SELF_CHECK, 1)
        for rep, n in enumerate(counts):
            h_bits, conf = synth.flat_tokens(w, n, 600 + rep)
            f = (h_bits.astype(np.uint32) << 16).view(np.float32).copy()
            f[1, ::3] *= 2.0 ** -12
            f[3, :] = 0.0
            f[5, :] *= 2.0 ** 6
            h_bits = (f.view(np.uint32) >> 16).astype(np.uint16)
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            outs = []
            with np.errstate(over="ignore"):
                ref = ora.denoise_step(0, h_bits, conf)
            for again, direct in enumerate((1, 1, 0)):
                run.ctx.set_option(binding.OPT_FP8_DIRECT, direct)
                out = torch.empty((n, h), dtype=torch.bfloat16, device=run.device)
                run.step(0, x, c, out)
                if again == 0:
                    _check_step(run, 0, n, out, ref, check_out=False)
                else:
                    ora.denoise_step(0, h_bits, conf)      # (keeps the oracle's resident set in step)
                outs.append(dev_to_bits(out))
            assert np.array_equal(outs[0], outs[1])
            got = [synth.bf16_bits_to_f32(o).astype(np.float64) for o in outs[1:]]
            rows = np.arange(n) != 5                       # (row 5 would be the whole norm)
            err = [np.linalg.norm((g - ref["out"])[rows]) / np.linalg.norm(ref["out"][rows]) for g in got]
            assert max(err) <= REL_L2 and err[0] <= 1.002 * err[1], err
            assert np.linalg.norm(got[0][5] - ref["out"][5]) <= REL_L2 * np.linalg.norm(ref["out"][5])
            assert np.all(got[0][3] == 0.0)
    finally:
        run.close()


def test_fp8_direct_form_takes_several_token_tiles_per_expert():
    """After a step in which no expert received more than 16 rows, the direct fp8 form's hit launch
    uses 16-row token tiles; a following step that sends all 24 tokens to the same two experts
    then needs two tiles per expert (the second one ragged)."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=8, top_k=2, hidden=256, intermediate=128)
    n = 24
    run = _runner(w, capacity=[8], max_tokens=n, fp8=True)
    ora = _oracle_for(run, [8])
    try:
        h_bits, conf = synth.flat_tokens(w, n, 52)
        same = np.repeat(h_bits[:1], n, axis=0)                  # every token the same row: one routing decision
        c = torch.from_numpy(conf).to(run.device)
        out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
        for rep, bits in enumerate((h_bits, h_bits, same, h_bits)):
            run.step(0, bits_to_dev(bits, run.device), c, out)
            ref = ora.denoise_step(0, bits, conf)
            if rep < 2:
                assert ref["counts"].max() <= 16
            if rep == 2:
                assert sorted(ref["counts"])[-2:] == [n, n]
            _check_step(run, 0, n, out, ref)
    finally:
        run.close()


def test_fp8_subnormal_codes_decode_exactly():
    """Blobs whose row scales are so large that every code is an e4m3 subnormal (exponent field
    0): the on-chip widening must reproduce them exactly, not flush them."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=4, top_k=2, hidden=256, intermediate=128)
    run = _runner(w, capacity=[4], max_tokens=24, fp8=True)
    try:
        h, i = w.hidden, w.intermediate
        rng = np.random.default_rng(77)
        for e in range(w.n_experts):
            blob = run.blobs[0][e]
            codes = (rng.integers(0, 8, size=3 * h * i).astype(np.uint8) |
                     (rng.integers(0, 2, size=3 * h * i).astype(np.uint8) << 7))     # +-{0..7} * 2^-9
            blob[:3 * h * i] = codes
            scales = rng.uniform(2.0, 6.0, size=2 * i + h).astype(np.float32)
            blob[3 * h * i:3 * h * i + 4 * scales.size] = scales.view(np.uint8)
        ora = _oracle_for(run, [4])
        h_bits, conf = synth.flat_tokens(w, 24, 60)
        x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
        out = torch.empty((24, h), dtype=torch.bfloat16, device=run.device)
        run.step(0, x, c, out)
        ref = ora.denoise_step(0, h_bits, conf)
        assert np.abs(ref["out"]).max() > 1e-3                 # the subnormal codes carry the whole signal
        _check_step(run, 0, 24, out, ref)
    finally:
        run.close()


def test_one_launch_and_two_launch_ffn_forms_agree_bit_for_bit():
    """OLED_OPT_FUSE_FFN: gate/up + down projection as one launch (down items wait on per-expert
    completion counters) or as two launches.  Which kernel computes an item does not change its
    arithmetic, so the layer outputs must be bit-identical, and both in parity with the oracle;
    token tiles of 16 to 128 rows, cold start so that launches of fetched experts (behind event
    waits) are covered too."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1, n_experts=6, top_k=3, hidden=512, intermediate=256)
    outs = {}
    for mode in (0, 2):
        run = _runner(w, capacity=[3], max_tokens=160)
        run.ctx.set_option(binding.OPT_FUSE_FFN, mode)
        ora = _oracle_for(run, [3])
        try:
            res = []
            for rep, n in enumerate((7, 33, 60, 150)):
                h_bits, conf = synth.flat_tokens(w, n, 80 + rep)
                x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
                out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
                run.step(0, x, c, out)
                _check_step(run, 0, n, out, ora.denoise_step(0, h_bits, conf))
                res.append(dev_to_bits(out).copy())
            outs[mode] = res
            _check_stats(run, ora)
        finally:
            run.close()
    for a, b in zip(outs[0], outs[2]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
@pytest.mark.parametrize("n_experts,top_k,hidden,inter", [(20, 3, 512, 384), (6, 6, 256, 128), (512, 2, 256, 128)])
def test_few_token_steps_at_the_edges_of_their_forms(n_experts, top_k, hidden, inter, fp8):
    """Steps of 1..32 tokens (every expert multiplies with the step's rows as they are), beyond (rows
    copied to their experts' regions; 512 experts x 65 tokens: too many, sorted rows), token tiles of 16 and
    32, weights loaded on the guess that the previous execution's experts return - right for a repeated
    input, wrong for the next one, where a run of nearly equal tokens leaves most experts without any."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=n_experts, top_k=top_k, hidden=hidden, intermediate=inter)
    run = _runner(w, capacity=[n_experts], max_tokens=65, fp8=fp8)
    ora = _oracle_for(run, [n_experts])
    try:
        for rep, n in enumerate((65, 32, 32, 17, 16, 1, 31, 33, 2, 64)):
            h_bits, conf = synth.flat_tokens(w, n, 200 + rep // 2)
            if rep % 3 == 1:
                h_bits[:] = h_bits[0]
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, x, c, out)
            _check_step(run, 0, n, out, ora.denoise_step(0, h_bits, conf))
        _check_stats(run, ora)
    finally:
        run.close()


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
@pytest.mark.parametrize("n_experts,top_k,inter,counts", [(4, 1, 128, (150, 200, 260, 520)), (10, 4, 128, (120, 130, 250)),
                                                           (512, 8, 128, (600,)), (64, 8, 1024, (250, 400, 512))])
def test_token_tiles_between_16_and_128_rows(n_experts, top_k, inter, counts, fp8):
    """Items of 48, 64, 96 and 128 token rows and several tiles per expert, with the tile taken from the previous
    execution's counts; 512 experts x 600 tokens: small tiles in a many-token step (bf16 outputs per assignment); 64 experts x 1024: more
    items than CTAs."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=n_experts, top_k=top_k, hidden=256, intermediate=inter)
    run = _runner(w, capacity=[n_experts], max_tokens=max(counts), fp8=fp8)
    ora = _oracle_for(run, [n_experts])
    try:
        for rep, n in enumerate(counts + counts[:1]):
            h_bits, conf = synth.flat_tokens(w, n, 300 + rep)
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, x, c, out)
            _check_step(run, 0, n, out, ora.denoise_step(0, h_bits, conf))
        _check_stats(run, ora)
    finally:
        run.close()


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
@pytest.mark.parametrize("n_experts,top_k,hidden,inter,n", [(8, 2, 512, 384, 40), (8, 2, 1024, 256, 148), (6, 3, 256, 128, 250),
                                                           (4, 1, 2048, 512, 290)])
def test_guess_rows_requested_before_the_counts(n_experts, top_k, hidden, inter, n, fp8):
    """Scattered steps whose guesses are right, wrong (equal tokens leave most experts without any) and right again, with
    one and two k-blocks per stage and items shorter and longer than the ring: the rows requested ahead are the item's."""
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1, n_experts=n_experts, top_k=top_k, hidden=hidden, intermediate=inter)
    run = _runner(w, capacity=[n_experts], max_tokens=n, fp8=fp8)
    ora = _oracle_for(run, [n_experts])
    try:
        for rep in range(5):
            h_bits, conf = synth.flat_tokens(w, n, 600 + rep // 2)
            if rep == 2:
                h_bits[:] = h_bits[0]
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, x, c, out)
            ref = ora.denoise_step(0, h_bits, conf)
            _check_step(run, 0, n, out, ref, check_out=False)
            got = synth.bf16_bits_to_f32(dev_to_bits(out)).astype(np.float64)
            # hidden 1024 and more give outputs beyond 4, where one rounding to bf16 is already 2^-9 of the value: that one and
            # those of the intermediate rows (2^-9 each, of a sum over them) stay below 2^-8 of the largest output
            assert np.abs(got - ref["out"]).max() <= max(MAX_ABS, 2.0 ** -8 * np.abs(ref["out"]).max())
            assert np.linalg.norm(got - ref["out"]) <= REL_L2 * np.linalg.norm(ref["out"])
        _check_stats(run, ora)
    finally:
        run.close()


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
@pytest.mark.parametrize("n", [20, 40, 250])
def test_the_rest_of_a_guess_called_ahead_changes_nothing(n, fp8):
    """Items several times longer than the ring, whose rest the counting warp (one launch) or the MMA warp (two) calls into L2
    until the gate is through - or not at all, where the launch does not start ahead of the gate (OLED_OPT_PDL 0): the same bits in
    all four forms for right and wrong guesses, and in parity with the oracle."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1, n_experts=8, top_k=2, hidden=4096, intermediate=128)
    outs = []
    for fuse, pdl in ((1, 1), (1, 0), (0, 1), (0, 0)):
        run = _runner(w, capacity=[8], max_tokens=n, fp8=fp8)
        run.ctx.set_option(binding.OPT_FUSE_FFN, fuse)
        run.ctx.set_option(binding.OPT_PDL, pdl)
        ora = _oracle_for(run, [8])
        try:
            for rep in range(4):
                h_bits, conf = synth.flat_tokens(w, n, 650)
                if rep == 2:
                    h_bits[:] = h_bits[0]
                x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
                out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
                run.step(0, x, c, out)
                outs.append(dev_to_bits(out).copy())
                if not outs[4:]:
                    ref = ora.denoise_step(0, h_bits, conf)
                    _check_step(run, 0, n, out, ref, check_out=False)
                    got = synth.bf16_bits_to_f32(outs[-1]).astype(np.float64)
                    # a rounding to bf16 moves a value by at most 2^-8 of it: the output's own, and those of the intermediate
                    # rows, whose sum is at most 2^-8 of an output's root mean square in standard deviation (six of them)
                    assert np.abs(got - ref["out"]).max() <= 2.0 ** -8 * (np.abs(ref["out"]).max() + 6.0 * np.sqrt(np.mean(ref["out"] ** 2)))
                    assert np.linalg.norm(got - ref["out"]) <= REL_L2 * np.linalg.norm(ref["out"])
                else:
                    assert np.array_equal(outs[-1], outs[len(outs) - 5])
        finally:
            run.close()


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
@pytest.mark.parametrize("n_experts,top_k,hidden,counts", [(64, 8, 2048, (1, 33, 149)), (3, 2, 256, (1, 149)), (33, 4, 4096, (2, 148)),
                                                           (8, 2, 16384, (1, 3)), (70, 8, 2048, (1, 150)), (512, 32, 1024, (1, 12)),
                                                           (16, 2, 768, (5, 600)), (64, 8, 1792, (1, 16, 17, 148)), (70, 8, 1024, (2, 148)),
                                                           (400, 4, 256, (3, 20)), (32, 4, 1024, (16, 149, 296))])
def test_gate_with_the_router_matrix_fetched_ahead(n_experts, top_k, hidden, counts, fp8):
    """Few-token gate: the router matrix on chip ahead of the input (in a stack's second layer, up to 16 tokens in the first one
    and in lone steps too) wholly in shared memory, with its last chunk or the last two in registers, in one and in several passes
    over the experts, for one and two tokens per CTA; and not fetched ahead, where it does not fit whole or four tokens share a CTA.
    Logits, ids, gate scores and order equal the oracle's bit for bit, in a stack iteration (where the combine runs in the same
    kernel) the same as layer by layer."""
    from oracle import moe_layer as oracle_moe
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=2, n_experts=n_experts, top_k=top_k, hidden=hidden, intermediate=128)
    run = _runner(w, capacity=[n_experts] * 2, max_tokens=max(counts), fp8=fp8, distinct_layers=1)
    try:
        for n in counts:
            h_bits, conf = synth.flat_tokens(w, n, 700)
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            out, nxt, both = (torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device) for _ in range(3))
            run.ctx.denoise_iteration(x.data_ptr(), c.data_ptr(), n, both.data_ptr())
            run.ctx.synchronize()
            for l in range(2):
                run.step(l, x, c, out)
                dbg = run.ctx.debug_last(l, n)
                logits = oracle_moe.gate_logits(oracle_moe.bf16_to_f32(dev_to_bits(x)),
                                                oracle_moe.bf16_to_f32(run.router_bits[l]), run.bias[l])
                ids, gate = oracle_moe.topk_route(logits, top_k)
                assert np.array_equal(run.ctx.debug_logits(l, n).view(np.uint32), logits.view(np.uint32))
                assert np.array_equal(dbg["ids"], ids)
                assert np.array_equal(dbg["gate"].view(np.uint32), gate.view(np.uint32))
                assert np.array_equal(dbg["perm"], oracle_moe.permutation(ids, n_experts)[2])
                run.ctx.residual_add(x.data_ptr(), out.data_ptr(), nxt.data_ptr(), x.numel())
                x, nxt = nxt, torch.empty_like(nxt)
            assert np.array_equal(dev_to_bits(x), dev_to_bits(both))
    finally:
        run.close()


@pytest.mark.parametrize("n_experts,top_k,counts", [(16, 16, (297, 1030)), (65, 14, (300, 2072)), (512, 32, (298, 401))])
def test_gate_sums_of_tokens_in_two_segments(n_experts, top_k, counts):
    """Many-token gate: a CTA's 8 to 14 tokens lie in one segment of the order or in two, segments are 20 tokens at the
    least, and tokens and experts end inside a tile; routing, order and reuse scores equal the oracle's."""
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=n_experts, top_k=top_k, hidden=256, intermediate=128)
    run = _runner(w, capacity=[n_experts], max_tokens=max(counts))
    ora = _oracle_for(run, [n_experts])
    try:
        for rep, n in enumerate(counts):
            h_bits, conf = synth.flat_tokens(w, n, 500 + rep)
            x, c = bits_to_dev(h_bits, run.device), torch.from_numpy(conf).to(run.device)
            out = torch.empty((n, w.hidden), dtype=torch.bfloat16, device=run.device)
            run.step(0, x, c, out)
            _check_step(run, 0, n, out, ora.denoise_step(0, h_bits, conf))
        _check_stats(run, ora)
    finally:
        run.close()


@pytest.mark.parametrize("n_experts,top_k,hidden", [(8, 3, 512), (64, 8, 2048), (512, 32, 256), (33, 1, 256)])
def test_routing_alone_at_the_edges_of_its_range(n_experts, top_k, hidden):
    """oled_route_noalloc from 1 to 256 tokens (one and two tokens per CTA, parts of the assignment list of one warp and
    of many), with a bias: ids, gate scores, counts, offsets and the stable order equal the oracle's bit for bit."""
    from oracle import moe_layer as oracle_moe
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev
    dev = torch.device("cuda:0")
    w = synth.tiny(n_layers=1, n_experts=n_experts, top_k=top_k, hidden=hidden, zipf_bias=0.3)
    wr_bits, bias = synth.router_weights(w, 0)
    wr, b = bits_to_dev(wr_bits, dev), torch.from_numpy(bias).to(dev)
    stream = torch.cuda.current_stream(dev).cuda_stream
    for n in (256, 1, 148, 149, 33, 255):
        h_bits, conf = synth.flat_tokens(w, n, 400)
        x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
        ids, perm = (torch.full((n * top_k,), -1, dtype=torch.int32, device=dev) for _ in range(2))
        gate = torch.zeros(n * top_k, device=dev)
        counts, offsets = (torch.full((m,), -1, dtype=torch.int32, device=dev) for m in (n_experts, n_experts + 1))
        rc = binding.route_noalloc(x.data_ptr(), wr.data_ptr(), b.data_ptr(), c.data_ptr(), n, hidden, n_experts, top_k, stream,
                                   ids.data_ptr(), gate.data_ptr(), counts.data_ptr(), offsets.data_ptr(), perm.data_ptr())
        assert rc == binding.OLED_OK, binding.strerror(rc)
        torch.cuda.synchronize(dev)
        logits = oracle_moe.gate_logits(oracle_moe.bf16_to_f32(h_bits), oracle_moe.bf16_to_f32(wr_bits), bias)
        o_ids, o_gate = oracle_moe.topk_route(logits, top_k)
        o_counts, o_offsets, o_perm, _ = oracle_moe.permutation(o_ids, n_experts)
        assert np.array_equal(ids.cpu().numpy().reshape(n, top_k), o_ids)
        assert np.array_equal(gate.cpu().numpy().view(np.uint32).reshape(n, top_k), o_gate.view(np.uint32))
        assert np.array_equal(counts.cpu().numpy(), o_counts) and np.array_equal(offsets.cpu().numpy(), o_offsets)
        assert np.array_equal(perm.cpu().numpy(), o_perm)


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
@pytest.mark.parametrize("n", [20, 40])
def test_contexts_on_streams_of_their_own_run_side_by_side(n, fp8):
    """Two contexts, each with a stream (of different priority) and a host thread of its own, next to matrix
    products on a third stream: the SMs a one-launch expert FFN gets, and when, are then up to the others.  No wait runs out
    and every iteration's output is, bit for bit, the one the context computes by itself; there are more gate/up
    items (24 experts x 8 weight tiles) than SMs, and half of the iterations meet other tokens than the one before."""
    import threading
    from paper_2609_33385_b200.runner import bits_to_dev
    w = synth.tiny(n_layers=4, n_experts=24, top_k=4, hidden=512, intermediate=512)
    iters, dev = 40, torch.device("cuda:0")
    a = torch.randn((4096, 4096), device=dev).to(torch.bfloat16)
    streams = [torch.cuda.Stream(dev, priority=0), torch.cuda.Stream(dev, priority=-1)]
    runs, inputs, alone, beside, errors = [], [], [], [], []
    try:
        for i, st in enumerate(streams):
            with torch.cuda.stream(st):
                runs.append(_runner(w, capacity=[24] * 4, max_tokens=n, fp8=fp8, share_store_of=runs[0] if runs else None))
            seeds = [300 + 10 * i + j // 2 % 3 for j in range(iters)]
            made = {s: synth.flat_tokens(w, n, s) for s in set(seeds)}
            made = {s: (bits_to_dev(x, dev), torch.from_numpy(c).to(dev)) for s, (x, c) in made.items()}
            inputs.append([made[s] for s in seeds])
            alone.append([torch.empty((n, w.hidden), dtype=torch.bfloat16, device=dev) for _ in seeds])
            beside.append([torch.empty((n, w.hidden), dtype=torch.bfloat16, device=dev) for _ in seeds])
        torch.cuda.synchronize(dev)

        def go(i, outs):
            try:
                torch.cuda.set_device(dev)
                for (x, c), out in zip(inputs[i], outs[i]):
                    runs[i].ctx.denoise_iteration(x.data_ptr(), c.data_ptr(), n, out.data_ptr())
                runs[i].ctx.synchronize()
            except Exception as e:                        # (shown by the main thread)
                errors.append(e)

        for i in range(2):
            go(i, alone)
        threads = [threading.Thread(target=go, args=(i, beside)) for i in range(2)]
        for t in threads:
            t.start()
        with torch.cuda.stream(torch.cuda.Stream(dev)):
            for _ in range(40):
                a @ a
        for t in threads:
            t.join()
        torch.cuda.synchronize(dev)
        assert not errors, errors
        for i in range(2):
            for x, y in zip(alone[i], beside[i]):
                assert torch.equal(x.view(torch.int16), y.view(torch.int16))
    finally:
        for r in runs:
            r.close()


@pytest.mark.parametrize("direct", [1, 0], ids=["direct", "widening"])
@pytest.mark.parametrize("n", [24, 300, 4200])
def test_fp8_intermediate_rows_that_overflow_give_no_finite_outputs(n, direct):
    """A token whose SwiGLU product exceeds the largest bf16 in one feature: its intermediate row holds an infinity, so every
    output the feature has a weight in is not finite, whatever form the codes are read in; the other tokens are unaffected.
    The down codes are the smallest there are (2^-9): a form that let the infinity saturate to a finite code would give
    ordinary numbers."""
    from paper_2609_33385_b200 import binding
    from paper_2609_33385_b200.runner import bits_to_dev, dev_to_bits
    w = synth.tiny(n_layers=1, n_experts=4, top_k=1, hidden=1024, intermediate=1024)
    run = _runner(w, capacity=[4], max_tokens=n, fp8=True)
    try:
        run.ctx.set_option(binding.OPT_FP8_DIRECT, direct)
        h, i, f = w.hidden, w.intermediate, 37
        for e in range(w.n_experts):
            blob = run.blobs[0][e]
            for m in (0, 1):                              # feature f, and no other, sees a row's first element: times 1.0
                codes = blob[m * i * h:(m + 1) * i * h].reshape(i, h)
                codes[:, 0] = 0
                codes[f] = 0
                codes[f, 0] = 0x38
            blob[2 * i * h:3 * i * h].reshape(h, i)[:, f] = 0x01
            scales = blob[3 * h * i:3 * h * i + 4 * (2 * i + h)].view(np.float32)
            scales[[f, i + f]] = 1.0
        h_bits, conf = synth.flat_tokens(w, n, 90)
        h_bits[:, 0] = 0x3F80
        c = torch.from_numpy(conf).to(run.device)
        outs = []
        for first in (0x3F80, 0x6280):                    # 1.0, then 2^70 in row 5: a product of 2^140
            h_bits[5, 0] = first
            out = torch.empty((n, h), dtype=torch.bfloat16, device=run.device)
            run.step(0, bits_to_dev(h_bits, run.device), c, out)
            run.ctx.synchronize()
            outs.append(dev_to_bits(out))
        finite = np.isfinite(synth.bf16_bits_to_f32(outs[1]))
        assert np.isfinite(synth.bf16_bits_to_f32(outs[0])).all()
        assert not finite[5].any()
        others = np.arange(n) != 5
        assert np.array_equal(outs[0][others], outs[1][others])
    finally:
        run.close()


@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
def test_a_context_that_fits_only_without_scatter_rows(fp8):
    """Device memory short of what few-token steps would like for a region of rows per expert (512 experts, 64 tokens: 32768
    rows instead of 64): the context is created all the same, its steps sort their rows, with the same outputs."""
    from paper_2609_33385_b200.runner import bits_to_dev
    n, e, h = 64, 512, 768
    w = synth.tiny(n_layers=1, n_experts=e, top_k=1, hidden=h, intermediate=128)
    dev = torch.device("cuda:0")
    h_bits, conf = synth.flat_tokens(w, n, 70)
    x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
    outs = [torch.empty((n, h), dtype=torch.bfloat16, device=dev) for _ in range(2)]
    roomy = tight = hold = None
    try:
        roomy = _runner(w, capacity=[e], max_tokens=n, fp8=fp8)
        roomy.step(0, x, c, outs[0])
        roomy.ctx.synchronize()
        before = torch.cuda.mem_get_info(dev)[0]           # (every kernel module is loaded by now)
        again = _runner(w, capacity=[e], max_tokens=n, fp8=fp8, share_store_of=roomy)
        roomy_bytes = before - torch.cuda.mem_get_info(dev)[0]
        again.close()
        torch.cuda.empty_cache()
        surplus = (32768 - n) * (h + 128) * 2 * (2 if fp8 else 1)
        assert roomy_bytes > surplus
        keep = roomy_bytes - surplus // 2
        hold = torch.empty(torch.cuda.mem_get_info(dev)[0] - keep, dtype=torch.uint8, device=dev)
        tight = _runner(w, capacity=[e], max_tokens=n, fp8=fp8, share_store_of=roomy)
        assert keep - torch.cuda.mem_get_info(dev)[0] < roomy_bytes - surplus * 3 // 4
        hold = None
        torch.cuda.empty_cache()
        for _ in range(2):                                 # fetched experts, then resident ones
            tight.step(0, x, c, outs[1])
            tight.ctx.synchronize()
            assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))
        a, b = roomy.ctx.debug_last(0, n), tight.ctx.debug_last(0, n)
        assert all(np.array_equal(a[k], b[k]) for k in ("ids", "perm", "counts", "scores"))
    finally:
        hold = None
        torch.cuda.empty_cache()
        for r in (roomy, tight):
            if r is not None:
                r.close()
