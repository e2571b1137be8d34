"""The layer call's choice of state passing, and packed outputs that are not cleared."""
import pytest
import torch

from paper_2606_06034_b200 import binding as gdn

FLAGS = gdn.GDN_FLAG_G_RAW | gdn.GDN_FLAG_LAYOUT_BTHD | gdn.GDN_FLAG_K_L2NORM


@pytest.mark.parametrize("segments,heads,first", [(3, 37, 43), (3, 38, 56), (4, 29, 35), (5, 21, 33), (6, 16, 34), (7, 13, 35), (8, 11, 36)])
def test_line_between_plain_and_segmented(segments, heads, first):
    assert not gdn._segments_pay(64 * (first - 1), 64, segments, heads)
    assert gdn._segments_pay(64 * first, 64, segments, heads)
    assert not gdn._segments_pay(64 * 100000, 64, 1, heads) and not gdn._segments_pay(0, 64, segments, heads)
    assert not gdn._segments_pay(64 * 32, 64, segments, heads)  # (the layer call does not ask up to there)


@pytest.mark.parametrize("bounds,T,whole", [([0, 5, 9], 9, True), ([0, 0, 9, 9], 9, True), ([0, 5], 9, False), ([1, 9], 9, False),
                                            ([], 4, False), ([0], 0, True)])
def test_rows_are_cleared_unless_every_one_is_written(bounds, T, whole, monkeypatch):
    made = []
    monkeypatch.setattr(torch, "zeros", lambda *a, _f=torch.zeros, **k: made.append("zeros") or _f(*a, **k))
    gdn._rows_like((T, 2, 4), torch.empty(0, dtype=torch.bfloat16), bounds, T)
    assert (made == []) == whole


def _inputs(T, H_k, H_v, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    return (r(1, T, H_k, 128).bfloat16(), r(1, T, H_k, 128).bfloat16(), r(1, T, H_v, 128).bfloat16(), torch.sigmoid(r(1, T, H_v)),
            -torch.nn.functional.softplus(r(1, T, H_v)), 0.3 * r(1, H_v, 128, 128))


@pytest.mark.gpu
@pytest.mark.parametrize("H_k,H_v,chunks", [(1, 2, 1), (1, 2, 2), (1, 2, 35), (1, 2, 36), (16, 32, 42), (16, 32, 43), (19, 38, 55), (19, 38, 56),
                                            (32, 64, 92)])
@pytest.mark.parametrize("with_state", [False, True])
def test_layer_on_both_sides_of_the_line(H_k, H_v, chunks, with_state):
    """Both forms compute the same chain; they differ by the fp32 re-association of the state recurrence (at most 2^-24 per
    token of decay-free carry, far below 1e-5 of the state) and, where that flips a rounding of the output, by one bf16 unit
    (2^-8) of single elements. The layer gives the bits of the form that the line asks for."""
    Q, K, V, beta, g, S = _inputs(64 * chunks, H_k, H_v, chunks)
    S = S if with_state else None
    O, Sn = gdn.gated_delta_layer(Q, K, V, beta, g, S_in=S)
    W, U, _ = gdn.chunk_prepare(K, V, beta, g, 64, flags=FLAGS | gdn.GDN_FLAG_W_GATED, want_tinv=False)
    Op, Sp = gdn.chunk_state_output(Q, K, W, U, g, 64, 128 ** -0.5, S, flags=FLAGS)
    Os, Ss = gdn.chunk_state_output_segmented(Q[0], K[0], W[0], U[0], g[0], 64, 128 ** -0.5, None if S is None else S[0], flags=FLAGS)
    assert gdn.gdn_device_status() == gdn.GDN_OK
    assert O.shape == V.shape and Sn.shape == (1, H_v, 128, 128)
    for o, s in ((Op, Sp), (Os[None], Ss[None])):
        assert (Sn - s).norm() <= 1e-5 * s.norm()
        assert (O.float() - o.float()).norm() <= 1e-3 * o.float().norm()
    segmented = gdn._segments_pay(64 * chunks, 64, int(gdn.load_library().gdn_chunk_state_segments(H_v)), H_v)
    o, s = (Os[None], Ss[None]) if segmented else (Op, Sp)
    assert torch.equal(O.view(torch.int16), o.view(torch.int16)) and torch.equal(Sn.view(torch.int32), s.view(torch.int32))


@pytest.mark.gpu
@pytest.mark.parametrize("H_v,chunks", [(2, 10), (2, 80), (32, 16), (32, 96), (64, 40), (64, 256)])
def test_the_line_is_on_the_right_side_of_the_clock(H_v, chunks):
    """Well off the line, on either side, the form that the layer takes is the faster one (8, 3 and 2 segments)."""
    Q, K, V, beta, g, _ = _inputs(64 * chunks, 1, H_v, chunks)
    W, U, _ = gdn.chunk_prepare(K, V, beta, g, 64, flags=FLAGS | gdn.GDN_FLAG_W_GATED, want_tinv=False)
    forms = (lambda: gdn.chunk_state_output(Q, K, W, U, g, 64, 1.0, flags=FLAGS),
             lambda: gdn.chunk_state_output_segmented(Q[0], K[0], W[0], U[0], g[0], 64, 1.0, flags=FLAGS))
    time = []
    for call in forms:
        runs = []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda._sleep(200000)  # (the launches are queued before the first one runs)
            a.record()
            for _ in range(8):
                call()
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        time.append(min(runs))
    segmented = gdn._segments_pay(64 * chunks, 64, int(gdn.load_library().gdn_chunk_state_segments(H_v)), H_v)
    assert time[segmented] < time[not segmented]


@pytest.mark.gpu
def test_packed_rows_without_a_sequence_stay_zero_and_the_others_keep_their_bits():
    T, extra = 200, 40
    Q, K, V, beta, g, _ = (x[0] for x in _inputs(T + extra, 1, 2, 3))
    cu = [0, 64, 65, 65, 190, T]
    whole = gdn.gated_delta_layer(*(x[:T].contiguous() for x in (Q, K, V, beta, g)), cu_seqlens=cu)
    torch.empty(1 << 22, device="cuda").fill_(float("nan"))  # (what an uncleared allocation would show)
    part = gdn.gated_delta_layer(Q, K, V, beta, g, cu_seqlens=cu)
    assert torch.equal(part[0][:T], whole[0]) and torch.equal(part[1], whole[1])
    assert torch.count_nonzero(part[0][T:]).item() == 0
    W, U, Tinv, cs, cl = gdn.chunk_prepare_varlen(K, V, beta, g, cu, 64, flags=FLAGS)
    assert torch.count_nonzero(W[T:]).item() == 0 and torch.count_nonzero(U[T:]).item() == 0
    assert cs.tolist() == [0, 64, 65, 129, 190] and cl.tolist() == [64, 1, 64, 61, 10]
    assert cs.dtype == cl.dtype == torch.int32 and cs.is_contiguous() and cl.is_contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("n_seq", [3, 256, 257])
def test_packed_sequences_taken_longest_first_keep_their_places(n_seq):
    """More runs than SMs: states and rows stay the ones of the single-sequence calls, bit for bit. Ties and empty sequences among
    them."""
    H_v = 64 if n_seq == 3 else 2
    gen = torch.Generator().manual_seed(n_seq)
    lens = torch.randint(0, 5, (n_seq,), generator=gen) * torch.randint(1, 40, (n_seq,), generator=gen)
    lens[0], lens[-1] = 3, 129
    cu = [0] + torch.cumsum(lens, 0).tolist()
    Q, K, V, beta, g, _ = (x[0] for x in _inputs(cu[-1], 1, H_v, n_seq))
    S0 = 0.3 * torch.randn(n_seq, H_v, 128, 128, generator=gen).cuda()
    O, S = gdn.gated_delta_layer(Q, K, V, beta, g, cu_seqlens=cu, S_in=S0)
    assert gdn.gdn_device_status() == gdn.GDN_OK
    for s in sorted({0, 1, 2, n_seq // 2, n_seq - 2, n_seq - 1, int(lens.argmax()), int(lens.argmin())}):
        a, b = cu[s], cu[s + 1]
        if a == b:
            assert torch.equal(S[s], S0[s])
            continue
        o, st = gdn.gated_delta_layer(*(x[a:b].clone() for x in (Q, K, V, beta, g)), cu_seqlens=[0, b - a], S_in=S0[s:s + 1].clone())
        assert torch.equal(O[a:b], o) and torch.equal(S[s], st[0])


@pytest.mark.gpu
@pytest.mark.parametrize("n_seq,H_v", [(2, 128), (60, 4), (64, 4), (65, 4), (128, 2), (129, 2), (256, 1), (257, 1), (512, 1)])
def test_longest_first_gives_what_the_order_of_arrival_gives(n_seq, H_v):
    """The forms for up to 64, 128, 256 and 512 sequences, on lengths for which the order is used, against the same sequences with
    empty ones behind them, too many for it: the same bits. Lengths at the edges of the classes, ties, empty sequences, one longer
    than the last class."""
    gen = torch.Generator().manual_seed(n_seq)
    lens = (64 * torch.exp(1.5 * torch.randn(n_seq, generator=gen) + 1.0)).int() % 4000
    lens[::7] = 64 * torch.randint(0, 14, lens[::7].shape, generator=gen).int()
    lens[n_seq // 2] = 64 * 500 + 1
    cu = [0] + torch.cumsum(lens, 0).tolist()
    chunks = cu[-1] / 64 + n_seq / 2
    assert n_seq * H_v > 148 and n_seq * H_v * n_seq * (125 + n_seq) <= 750 * 148 * chunks
    Q, K, V, beta, g, _ = (x[0] for x in _inputs(cu[-1], 1, H_v, n_seq))
    S0 = 0.3 * torch.randn(513, H_v, 128, 128, generator=gen).cuda()
    W, U, _, _, _ = gdn.chunk_prepare_varlen(K, V, beta, g, cu, 64, flags=FLAGS | gdn.GDN_FLAG_W_GATED, want_tinv=False)
    for flags in (FLAGS, FLAGS & ~gdn.GDN_FLAG_K_L2NORM):
        scale = 128 ** -0.5 if flags == FLAGS else 0.01
        O, S = gdn.chunk_state_output_varlen(Q, K, W, U, g, cu, 64, scale, S0[:n_seq].contiguous(), flags=flags)
        On, Sn = gdn.chunk_state_output_varlen(Q, K, W, U, g, cu + [cu[-1]] * (513 - n_seq), 64, scale, S0, flags=flags)
        assert gdn.gdn_device_status() == gdn.GDN_OK
        assert torch.equal(O.view(torch.int16), On.view(torch.int16)) and torch.equal(S.view(torch.int32), Sn[:n_seq].view(torch.int32))
        assert torch.equal(Sn[n_seq:], S0[n_seq:])


@pytest.mark.gpu
@pytest.mark.parametrize("B,H_k,H_v,chunks", [(1, 1, 1, 1), (1, 2, 6, 3), (2, 3, 3, 5), (3, 16, 32, 2)])
@pytest.mark.parametrize("token_major", [False, True])
def test_one_native_call_gives_what_the_two_calls_give(B, H_k, H_v, chunks, token_major):
    """Same kernels on the same inputs: the same bits, with and without a state carried in or asked for; and the argument errors of
    the two calls."""
    T = 64 * chunks
    gen = torch.Generator(device="cuda").manual_seed(B + H_v)
    r = lambda H, *d: torch.randn(*((B, T, H) if token_major else (B, H, T)), *d, generator=gen, device="cuda")
    Q, K, V = r(H_k, 128).bfloat16(), r(H_k, 128).bfloat16(), r(H_v, 128).bfloat16()
    beta, g, S0 = torch.sigmoid(r(H_v)), -torch.nn.functional.softplus(r(H_v)), 0.3 * torch.randn(B, H_v, 128, 128, generator=gen, device="cuda")
    flags = gdn.GDN_FLAG_G_RAW | gdn.GDN_FLAG_K_L2NORM | (gdn.GDN_FLAG_LAYOUT_BTHD if token_major else 0)
    W, U, _ = gdn.chunk_prepare(K, V, beta, g, 64, flags=flags | gdn.GDN_FLAG_W_GATED, want_tinv=False)
    for S, want in ((None, True), (S0, True), (S0, False)):
        O, Sn = gdn.gated_delta_layer(Q, K, V, beta, g, S_in=S, token_major=token_major, want_state=want)
        Op, Sp = gdn.chunk_state_output(Q, K, W, U, g, 64, 128 ** -0.5, S, want_state=want, flags=flags)
        assert gdn.gdn_device_status() == gdn.GDN_OK
        assert torch.equal(O.view(torch.int16), Op.view(torch.int16)) and (Sn is None) == (Sp is None) == (not want)
        assert Sn is None or torch.equal(Sn.view(torch.int32), Sp.view(torch.int32))
    with pytest.raises(gdn.GdnError):
        gdn.gated_delta_layer(Q, K, V, beta, g, C=32, token_major=token_major)
    for C in (0, -64):
        with pytest.raises(gdn.GdnError) as e:
            gdn.gated_delta_layer(Q, K, V, beta, g, C=C, token_major=token_major)
        assert e.value.status == gdn.GDN_ERR_INVALID_ARG
    with pytest.raises(ValueError):
        gdn.gated_delta_layer(torch.stack((Q, Q), -1)[..., 0], K, V, beta, g, token_major=token_major)


@pytest.mark.gpu
@pytest.mark.parametrize("B,H_k,H_v,chunks,with_state", [(1, 16, 32, 1, True), (3, 2, 4, 5, False), (8, 16, 32, 3, True), (1, 1, 2, 40, True)])
def test_layer_call_can_be_captured_and_replayed_on_new_inputs(B, H_k, H_v, chunks, with_state):
    """The native call (its second launch is a programmatic edge of the graph) and the segmented form: what the replay writes are
    the bits of a call outside of a graph, for the inputs captured and for others in their place."""
    def inputs(seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        r = lambda *s: torch.randn(*s, generator=gen, device="cuda")
        T = 64 * chunks
        return [r(B, T, H_k, 128).bfloat16(), r(B, T, H_k, 128).bfloat16(), r(B, T, H_v, 128).bfloat16(), torch.sigmoid(r(B, T, H_v)),
                -torch.nn.functional.softplus(r(B, T, H_v))] + ([0.3 * r(B, H_v, 128, 128)] if with_state else [])

    x = inputs(1)
    call = lambda t: gdn.gated_delta_layer(*t[:5], S_in=t[5] if with_state else None)
    want = [[y.clone() for y in call(inputs(seed))] for seed in (1, 2, 3)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        O, S = call(x)
    for seed in (1, 2, 3):
        for a, b in zip(x, inputs(seed)):
            a.copy_(b)
        graph.replay()
        graph.replay()
        assert torch.equal(O.view(torch.int16), want[seed - 1][0].view(torch.int16))
        assert torch.equal(S.view(torch.int32), want[seed - 1][1].view(torch.int32))
    assert gdn.gdn_device_status() == gdn.GDN_OK


@pytest.mark.gpu
@pytest.mark.parametrize("B,H_k,H_v,T,cu", [(1, 16, 32, 4096, None), (8, 32, 32, 1024, None), (1, 16, 32, 64, None),
                                            (1, 16, 32, 4111, [0, 5, 69, 700, 701, 1725, 2000, 3999, 4111])])
def test_repeated_layer_calls_are_bit_identical(B, H_k, H_v, T, cu):
    """No atomics on data and a fixed order of every sum, in the state passing too: repeated calls agree bit for bit, also while
    another stream keeps the memory system busy."""
    gen = torch.Generator(device="cuda").manual_seed(T)
    r = lambda *s: torch.randn(*(s if cu is None else s[1:]), generator=gen, device="cuda")
    args = (r(B, T, H_k, 128).bfloat16(), r(B, T, H_k, 128).bfloat16(), r(B, T, H_v, 128).bfloat16(), torch.sigmoid(r(B, T, H_v)),
            -torch.nn.functional.softplus(r(B, T, H_v)))
    ref = gdn.gated_delta_layer(*args, cu_seqlens=cu)
    assert gdn.gdn_device_status() == gdn.GDN_OK
    side, junk = torch.cuda.Stream(), torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    for rep in range(8):
        if rep % 2 == 1:
            with torch.cuda.stream(side):
                for _ in range(8):
                    junk.add_(1)
        O, S = gdn.gated_delta_layer(*args, cu_seqlens=cu)
        assert torch.equal(O.view(torch.int16), ref[0].view(torch.int16)) and torch.equal(S.view(torch.int32), ref[1].view(torch.int32))
    torch.cuda.synchronize()
    assert gdn.gdn_device_status() == gdn.GDN_OK
