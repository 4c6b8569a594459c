"""The allocation-free routing entry point against the regular step.

Some hosts hand all device memory to their own arena, or cannot afford the device-wide
synchronisation of cudaMalloc inside the decode loop; for them the library offers
``oled_route_noalloc``, which has no scratch at all.  The first test calls it
through the C ABI twice in a row, with different inputs (so stale contents of anything shared
would show), and checks every output bit for bit against what ``oled_denoise_step`` produced
for the same inputs and against the CPU oracle's gate, top-k and permutation of the same bits; the
second one overlaps calls on two streams.  They are collected last on purpose: a run that stops at the first
failure has then already run every other test.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import moe_layer as oracle_moe  # noqa: E402
from paper_2609_33385_b200 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def test_route_noalloc_matches_denoise_step_twice_in_a_row():
    from paper_2609_33385_b200 import binding, build
    build.build()
    from paper_2609_33385_b200.runner import StackRunner, bits_to_dev
    w = synth.tiny(n_layers=1, n_experts=8, top_k=3, hidden=512)
    run = StackRunner(w, capacity=[4], max_tokens=64)
    dev = run.device
    e, k, h = w.n_experts, w.top_k, w.hidden
    wr_dev, _ = run._router_dev[0]
    stream = torch.cuda.current_stream(dev).cuda_stream
    try:
        for call, n in enumerate((37, 9)):                # second call is smaller: stale rows would show
            h_bits, conf = synth.flat_tokens(w, n, 40 + call)
            x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
            out = torch.empty((n, h), dtype=torch.bfloat16, device=dev)
            run.step(0, x, c, out)
            ref = run.ctx.debug_last(0, n)

            ids = torch.full((n * k,), -1, dtype=torch.int32, device=dev)
            gate = torch.full((n * k,), -1.0, dtype=torch.float32, device=dev)
            counts = torch.full((e,), -1, dtype=torch.int32, device=dev)
            offsets = torch.full((e + 1,), -1, dtype=torch.int32, device=dev)
            perm = torch.full((n * k,), -1, dtype=torch.int32, device=dev)
            rc = binding.route_noalloc(x.data_ptr(), wr_dev.data_ptr(), None, c.data_ptr(), n, h, e, k,
                                       stream, ids.data_ptr(), gate.data_ptr(), counts.data_ptr(),
                                       offsets.data_ptr(), perm.data_ptr())
            assert rc == binding.OLED_OK, binding.strerror(rc)
            torch.cuda.synchronize(dev)
            assert np.array_equal(ids.cpu().numpy().reshape(n, k), ref["ids"])
            assert np.array_equal(gate.cpu().numpy().view(np.uint32).reshape(n, k),
                                  ref["gate"].view(np.uint32))            # same kernels: bit-exact
            assert np.array_equal(counts.cpu().numpy(), ref["counts"])
            assert np.array_equal(perm.cpu().numpy(), ref["perm"])
            off = offsets.cpu().numpy()
            assert off[0] == 0 and np.array_equal(np.diff(off), ref["counts"])
            # ... and against the oracle (independent of the CUDA path) on the same input bits
            logits = oracle_moe.gate_logits(oracle_moe.bf16_to_f32(h_bits),
                                            oracle_moe.bf16_to_f32(run.router_bits[0]), None)
            o_ids, o_gate = oracle_moe.topk_route(logits, k)
            o_counts, o_offsets, o_perm, _ = oracle_moe.permutation(o_ids, e)
            assert np.array_equal(ids.cpu().numpy().reshape(n, k), o_ids)
            assert np.array_equal(gate.cpu().numpy().view(np.uint32).reshape(n, k), o_gate.view(np.uint32))
            assert np.array_equal(counts.cpu().numpy(), o_counts)
            assert np.array_equal(off, o_offsets)
            assert np.array_equal(perm.cpu().numpy(), o_perm)
        # beyond the stated maximum: a clear error, nothing launched
        big = binding.NOALLOC_MAX_TOKENS + 1
        rc = binding.route_noalloc(x.data_ptr(), wr_dev.data_ptr(), None, c.data_ptr(), big, h, e, k,
                                   stream, ids.data_ptr(), gate.data_ptr(), counts.data_ptr(),
                                   offsets.data_ptr(), perm.data_ptr())
        assert rc == binding.ERR_TOO_MANY_TOKENS
    finally:
        run.close()


def test_overlapping_and_replayed_calls_share_nothing():
    """Calls that overlap on two streams, more than 1024 enqueued calls apart or side by side, and calls captured in a
    graph that is replayed next to live ones: every call's arrays hold what a call by itself gives."""
    from paper_2609_33385_b200 import binding, build
    build.build()
    from paper_2609_33385_b200.runner import bits_to_dev
    dev = torch.device("cuda:0")
    h, e, k, n = 512, 16, 3, 64
    w = synth.tiny(n_layers=1, n_experts=e, top_k=k, hidden=h)
    wr = bits_to_dev(synth.router_weights(w, 0)[0], dev)
    h_bits, conf = synth.flat_tokens(w, n, 60)
    x, c = bits_to_dev(h_bits, dev), torch.from_numpy(conf).to(dev)
    words = 3 * n * k + e + (e + 1)                       # ids, gate, perm, counts, offsets: one block per call
    words = (words + 3) // 4 * 4
    calls = 1100
    a, b = torch.cuda.Stream(dev), torch.cuda.Stream(dev)

    def call(block, stream):
        p = block.data_ptr()
        rc = binding.route_noalloc(x.data_ptr(), wr.data_ptr(), None, c.data_ptr(), n, h, e, k, stream.cuda_stream, p,
                                   p + 4 * n * k, p + 12 * n * k, p + 12 * n * k + 4 * e, p + 8 * n * k)
        assert rc == binding.OLED_OK, binding.strerror(rc)

    one = torch.zeros(words, dtype=torch.int32, device=dev)
    call(one, torch.cuda.current_stream(dev))
    torch.cuda.synchronize(dev)
    want = one.clone()
    assert int(want[3 * n * k:3 * n * k + e].sum()) == n * k
    for _ in range(3):
        blocks = torch.full((calls, words), -1, dtype=torch.int32, device=dev)
        blocks[:, 3 * n * k + e + (e + 1):] = want[3 * n * k + e + (e + 1):]
        first = torch.full((8, words), -1, dtype=torch.int32, device=dev)
        first[:, 3 * n * k + e + (e + 1):] = want[3 * n * k + e + (e + 1):]
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize(dev)
        with torch.cuda.graph(graph, stream=a):
            for i in range(4):
                call(first[i], a)
        torch.cuda.synchronize(dev)
        started = torch.cuda.Event()
        with torch.cuda.stream(b):
            torch.cuda._sleep(20_000_000)                 # (about ten milliseconds: the calls below queue up behind it)
            started.record(b)
        a.wait_event(started)
        for i in range(4, 8):                             # these run beside the calls on the other stream
            call(first[i], a)
        with torch.cuda.stream(a):
            graph.replay()
        for i in range(calls):
            call(blocks[i], b)
            if i % 100 == 0:
                with torch.cuda.stream(a):
                    graph.replay()
        torch.cuda.synchronize(dev)
        del graph
        assert bool((first == want).all()), "a call beside the others, or a captured one"
        assert bool((blocks == want).all()), "one of many calls on a stream"
