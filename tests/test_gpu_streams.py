"""The library enqueues on the caller's stream and allocates nothing: the whole path runs on a side stream and
inside a captured CUDA graph, with the same bits as on the default stream."""
import pytest
import torch

from paper_2505_07004_b200 import api as libgq
from paper_2505_07004_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


def make(dev):
    cfg = synth.LayerConfig("s", 1024 + 200, 512, 520, 64, (2,), "lognormal", 0.02, 20.0)
    syn = synth.LayerSynth(cfg, dev, seed=11)
    xs = [syn.x_chunk(c) for c in range(cfg.n_chunks)]
    gs = [syn.grad_chunk(c) for c in range(cfg.n_chunks)]
    W, What = syn.weights()
    return cfg, xs, gs, W, What


def run_path(cfg, xs, gs, W, What, bufs):
    H, s_buf, ws, ows, loss = bufs
    g = cfg.g
    H.zero_()
    for x, gr in zip(xs, gs):
        nt = x.shape[0]
        libgq.gq_saliency_prepared(gr, g, ws, 1.0, s=s_buf[:, :nt])
        libgq.gq_hessian_accumulate(x, s_buf[:, :nt], H, ws,
                                    flags=libgq.GQ_HESSIAN_DETERMINISTIC | libgq.GQ_HESSIAN_S_PREPARED)
    libgq.gq_hessian_finalize(H)
    libgq.gq_objective(W, What, H, ows, loss=loss)


def buffers(cfg, dev):
    g = cfg.g
    return (torch.empty(g, cfg.d_in, cfg.d_in, device=dev), torch.empty(g, cfg.chunk, device=dev),
            libgq.alloc_workspace(libgq.gq_hessian_workspace_bytes(cfg.chunk, cfg.d_in, g), dev),
            libgq.alloc_workspace(libgq.gq_objective_workspace_bytes(cfg.d_in, cfg.d_out, g), dev),
            torch.empty(g + 1, dtype=torch.float64, device=dev))


def test_side_stream_and_graph_replay_match_the_default_stream(dev):
    cfg, xs, gs, W, What = make(dev)
    ref = buffers(cfg, dev)
    run_path(cfg, xs, gs, W, What, ref)
    torch.cuda.synchronize()
    libgq.gq_check()

    side = torch.cuda.Stream()
    b1 = buffers(cfg, dev)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        run_path(cfg, xs, gs, W, What, b1)
    side.synchronize()
    libgq.gq_check()
    assert torch.equal(b1[0], ref[0]) and torch.equal(b1[4], ref[4])

    b2 = buffers(cfg, dev)
    graph = torch.cuda.CUDAGraph()
    launches0 = libgq.gq_launch_count()
    with torch.cuda.graph(graph):
        run_path(cfg, xs, gs, W, What, b2)
    per_step = libgq.gq_launch_count() - launches0
    assert per_step == 2 * cfg.n_chunks + 5          # saliency, Hessian per chunk; mirror, maximum, fp16, dot, reduce
    for _ in range(2):
        b2[0].fill_(7.0)
        b2[4].zero_()
        graph.replay()
    torch.cuda.synchronize()
    libgq.gq_check()
    assert torch.equal(b2[0], ref[0]) and torch.equal(b2[4], ref[4])


def run_path_ahead(cfg, xs, gs, W, What, bufs, extra):
    """The same path with one launch per chunk: the saliency of chunk c + 1 is computed inside the Hessian launch
    of chunk c (two saliency buffers and scratch blocks in turn)."""
    H, s_buf, ws, ows, loss = bufs
    sb, wb = (s_buf, extra[0]), (ws, extra[1])
    g = cfg.g
    flags = libgq.GQ_HESSIAN_DETERMINISTIC | libgq.GQ_HESSIAN_S_PREPARED
    H.zero_()
    libgq.gq_saliency_prepared(gs[0], g, wb[0], 1.0, s=sb[0][:, :gs[0].shape[0]])
    for c, x in enumerate(xs):
        nt = x.shape[0]
        if c + 1 < len(xs):
            libgq.gq_hessian_accumulate_ahead(x, sb[c & 1][:, :nt], H, wb[c & 1], gs[c + 1], wb[(c + 1) & 1], 1.0,
                                              sb[(c + 1) & 1][:, :gs[c + 1].shape[0]], flags=flags)
        else:
            libgq.gq_hessian_accumulate(x, sb[c & 1][:, :nt], H, wb[c & 1], flags=flags)
    libgq.gq_hessian_finalize(H)
    libgq.gq_objective(W, What, H, ows, loss=loss)


def test_one_launch_per_chunk_in_a_graph_gives_the_same_bits(dev):
    cfg, xs, gs, W, What = make(dev)
    assert cfg.n_chunks >= 3
    ref = buffers(cfg, dev)
    run_path(cfg, xs, gs, W, What, ref)
    torch.cuda.synchronize()
    b = buffers(cfg, dev)
    extra = (torch.empty_like(b[1]), libgq.alloc_workspace(libgq.gq_hessian_workspace_bytes(cfg.chunk, cfg.d_in, cfg.g), dev))
    graph = torch.cuda.CUDAGraph()
    launches0 = libgq.gq_launch_count()
    with torch.cuda.graph(graph):
        run_path_ahead(cfg, xs, gs, W, What, b, extra)
    assert libgq.gq_launch_count() - launches0 == cfg.n_chunks + 1 + 5
    for _ in range(2):
        b[0].fill_(7.0)
        b[4].zero_()
        graph.replay()
    torch.cuda.synchronize()
    libgq.gq_check()
    assert torch.equal(b[0], ref[0]) and torch.equal(b[4], ref[4])


def test_steps_enqueued_without_a_pause_read_what_the_step_before_wrote(dev):
    """Kernels start before the ones they follow have ended.  Layers small enough for a kernel and the next ones to be on
    the GPU at the same time: quantiser, objective, Hessian and finalize again and again over the same buffers, without a
    pause and with one after every call, give the same values.  (Descent adds its panel pieces in any order, so a decision
    may differ where two levels are equally near, to 1e-6 of the target; that changes the objective by far less than 1e-4.
    A buffer of the round before holds other inputs, whose objective is percents away.)"""
    m, g, d_in, d_out, n = 4, 2, 264, 64, 200
    gen = torch.Generator(device=dev).manual_seed(3)
    cases = []
    for _ in range(3):
        X = torch.randn(n, d_in, generator=gen, device=dev).to(torch.bfloat16)
        W = 0.02 * torch.randn(d_out, d_in, generator=gen, device=dev)
        cb = torch.quantile(W, (torch.arange(m, device=dev) + 0.5) / m, dim=1).T.contiguous()
        cases.append((X, torch.rand(g, n, generator=gen, device=dev), W, cb))

    def run(pause):
        H, What = torch.empty(g, d_in, d_in, device=dev), torch.empty(d_out, d_in, device=dev)
        loss = torch.empty(30, g + 1, dtype=torch.float64, device=dev)
        hws = libgq.alloc_workspace(libgq.gq_hessian_workspace_bytes(n, d_in, g), dev)
        cws = libgq.alloc_workspace(libgq.gq_cd_workspace_bytes(d_in, d_out, g), dev)
        ows = libgq.alloc_workspace(libgq.gq_objective_workspace_bytes(d_in, d_out, g), dev)
        for i in range(30):
            X, s, W, cb = cases[i % 3]
            for step in (lambda: H.zero_(),
                         lambda: libgq.gq_hessian_accumulate(X, s, H, hws, flags=libgq.GQ_HESSIAN_DETERMINISTIC),
                         lambda: libgq.gq_hessian_finalize(H),
                         lambda: What.copy_(cb[:, :1].expand(-1, d_in)),
                         lambda: libgq.gq_cd_cycles(W, What, cb, H, 1, cws),
                         lambda: libgq.gq_objective(W, What, H, ows, loss=loss[i])):
                step()
                if pause:
                    torch.cuda.synchronize()
        libgq.gq_check()
        return loss

    paused = run(True)
    assert ((paused[0] - paused[1]).abs() > 1e-3 * paused[0]).all() and ((paused[1] - paused[2]).abs() > 1e-3 * paused[1]).all()
    torch.testing.assert_close(run(False), paused, rtol=1e-4, atol=0.0)


def test_two_streams_at_once(dev):
    """Two chains of calls in flight on two streams, each with its own buffers: the same bits as alone."""
    cfg, xs, gs, W, What = make(dev)
    ref = buffers(cfg, dev)
    run_path(cfg, xs, gs, W, What, ref)
    torch.cuda.synchronize()
    sides = [(torch.cuda.Stream(), buffers(cfg, dev)) for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(20):
        for st, b in sides:
            with torch.cuda.stream(st):
                run_path(cfg, xs, gs, W, What, b)
    torch.cuda.synchronize()
    libgq.gq_check()
    for _, b in sides:
        assert torch.equal(b[0], ref[0]) and torch.equal(b[4], ref[4])


def test_quantiser_in_a_graph(dev):
    """gq_cd_cycles and gq_lnq captured and replayed twice, against the same calls outside.  One block of coordinates:
    descent has no panel pieces whose order could vary; the codebooks' fp64 sums do, in their last bits."""
    m, g, d, d_out = 8, 2, 256, 96
    gen = torch.Generator(device=dev).manual_seed(8)
    X = torch.randn(2 * d, d, generator=gen, device=dev)
    H = (X.T @ X).expand(g, d, d).contiguous()
    H = ((H + H.transpose(1, 2)) / 2).contiguous()
    W = 0.02 * torch.randn(d_out, d, generator=gen, device=dev)
    cb0 = torch.quantile(W, (torch.arange(m, device=dev) + 0.5) / m, dim=1).T.contiguous()
    Q0 = (W[:, :, None] - cb0[:, None, :]).abs().argmin(2).to(torch.uint8)
    W0 = torch.gather(cb0, 1, Q0.long())
    cws = libgq.alloc_workspace(libgq.gq_cd_workspace_bytes(d, d_out, g), dev)
    lws = libgq.alloc_workspace(libgq.gq_lnq_workspace_bytes(d, d_out, g, m), dev)
    W_cd, Q_cd, Q_lnq = torch.empty_like(W), torch.empty_like(Q0), torch.empty_like(Q0)

    def both():
        W_cd.copy_(W0)
        Q_lnq.copy_(Q0)
        libgq.gq_cd_cycles(W, W_cd, cb0, H, 2, cws, Q=Q_cd)
        return libgq.gq_lnq(W, Q_lnq, m, H, 2, 2, lws)

    W_l, _, cb_l = both()
    want = [t.clone() for t in (W_cd, Q_cd, Q_lnq, W_l, cb_l)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        W_l, _, cb_l = both()
    for _ in range(2):
        for t in (W_cd, Q_cd, Q_lnq, W_l, cb_l):
            t.fill_(1)
        graph.replay()
    torch.cuda.synchronize()
    libgq.gq_check()
    assert torch.equal(W_cd, want[0]) and torch.equal(Q_cd, want[1])
    assert (Q_lnq != want[2]).float().mean() <= 0.01
    same = (Q_lnq == want[2]).all(1)
    torch.testing.assert_close(cb_l[same], want[4][same], rtol=1e-5, atol=1e-6)
    torch.testing.assert_close(W_l[same], want[3][same], rtol=1e-5, atol=1e-6)
