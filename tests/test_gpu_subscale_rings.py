"""Subscale generation through the conditioning network as one staggered schedule on rings, network and stepping side by side."""
import numpy as np
import pytest

from oracle import subscale_net as sn
from oracle import wrnn_oracle as orc
from paper_1802_08435_b200 import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

SEED, F = synth.SEED_SAMPLING, 128


# even and odd numbers of rows (a tile has two), lengths that are no multiple of a block of 64, a row that ends inside the block in which others go on,
# gaps between rows (lag > L) of one, two and five blocks, k-blocks shared by one, two and three CTAs (rows, taps), a network without reach
@pytest.mark.parametrize("rows,L,chunk,lag,net", [
    (16, 300, 128, 256, dict()), (3, 700, 64, 256, dict()), (5, 130, 128, 384, dict()), (2, 20, 64, 512, dict()), (2, 64, 128, 256, dict()),
    (12, 420, 128, 384, dict(dilations=(1, 5, 32))), (3, 200, 64, 256, dict(taps=2, dilations=(64, 9))), (4, 150, 128, 256, dict(taps=1, dilations=(1, 1))),
    (3, 190, 64, 256, dict(taps=4, dilations=(7, 21, 11), conv_ch=192, res_ch=384)), (20, 150, 64, 256, dict(dilations=(2, 2)))])
def test_rings(rows, L, chunk, lag, net):
    """Every draw against the oracle forced on the device's samples; chunks of 32 go through the calls one by one, without rings, and draw the
    same but for near-boundary draws; a second call, one on another stream and a replayed capture of one draw exactly the same."""
    import torch
    from paper_1802_08435_b200 import binding as B
    w, nw = synth.make_weights(896, cond_dim=synth.COND_DIM), synth.make_subscale_net(rows, **net)
    frames = synth.make_cond(rows, rows * L // synth.HOP + 2, synth.COND_DIM)
    f_d = torch.from_numpy(frames).cuda()
    m, q = B.wrnn_create(w, "bf16", max_batch=rows), B.wrnn_subscale_net_create(nw)

    def call(out, ch=chunk, lg=lag, stream=None):
        B.wrnn_sample_subscale_net(m, q, f_d, F, ch, lg, rows * L, SEED, out, stream=stream)

    def run(**kw):
        out = torch.zeros(rows * L, dtype=torch.int16, device="cuda:0")
        call(out, **kw)
        torch.cuda.synchronize()
        assert B.wrnn_poll_status(m) == 0 and B.wrnn_subscale_net_status(q) == 0
        return out.cpu().numpy()

    try:
        out = run()
        got = orc.fold(out, rows)
        want, _, mg = sn.subscale_net_run(orc.OracleModel(w, "bf16"), sn.SubscaleNet(nw), frames, L, synth.HOP, SEED, forced=got, teacher=True)
        for g, r, k in zip(pu._split(got), pu._split(want), (0, 1)):
            assert pu.check_indices(g, r, mg[:, :, k])[1] == 0
        one_by_one = run(ch=32, lg=256)
        assert (one_by_one != out).mean() <= max(2e-3, 2.5 / out.size)
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            assert np.array_equal(run(stream=side), out) and np.array_equal(run(), out)
        graph, cap = torch.cuda.CUDAGraph(), torch.zeros(rows * L, dtype=torch.int16, device="cuda:0")
        with torch.cuda.graph(graph):
            call(cap)
        cap.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(cap.cpu().numpy(), out)
        del graph
    finally:
        B.wrnn_subscale_net_destroy(q)
        B.wrnn_destroy(m)


@pytest.mark.parametrize("chunk", [64, 32])
def test_first_call_of_a_network_on_a_stream_of_its_own(chunk):
    """A network makes its workspaces at its first call and clears them in the order of that call's stream: what waits on the default stream,
    with which the streams here do not block, neither holds the clearing back nor lets it fall into the call.  With rings and without."""
    import torch
    from paper_1802_08435_b200 import binding as B
    rows, L = 6, 900
    nw = synth.make_subscale_net(rows)
    frames = torch.from_numpy(synth.make_cond(rows, rows * L // synth.HOP + 2, synth.COND_DIM)).cuda()
    m = B.wrnn_create(synth.make_weights(896), "bf16", max_batch=rows)

    def first(stream, busy=0):
        q, out = B.wrnn_subscale_net_create(nw), torch.zeros(rows * L, dtype=torch.int16, device="cuda:0")
        try:
            torch.cuda.synchronize()
            if busy:
                torch.cuda._sleep(busy)
            B.wrnn_sample_subscale_net(m, q, frames, F, chunk, 256, rows * L, SEED, out, stream=stream)
            torch.cuda.synchronize()
            assert B.wrnn_poll_status(m) == 0 and B.wrnn_subscale_net_status(q) == 0
            return out.cpu().numpy()
        finally:
            B.wrnn_subscale_net_destroy(q)

    try:
        want, side = first(None), torch.cuda.Stream()               # (the model's own workspaces are made here)
        for busy in (0, 1_000_000, 4_000_000, 10_000_000):          # clocks: up to 5 ms, half of a call
            assert np.array_equal(first(side, busy), want)
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("dtype,rows,conv_ch", [("bf16", 30, 192), ("f32", 12, 96)])
def test_rings_with_all_rows_under_way(dtype, rows, conv_ch):
    """Rows that follow one another closely enough for all of them to be under way at once: every count of rows per cluster, up to the kernel of many
    rows, and more clusters than the schedule leaves for the stepping otherwise.  The draws of rows spread over the schedule against the oracle
    forced on the device's samples."""
    import torch
    from concurrent.futures import ThreadPoolExecutor
    from paper_1802_08435_b200 import binding as B
    lag = 128
    L = lag * (rows - 1) + 90
    w, nw = synth.make_weights(896), synth.make_subscale_net(rows, conv_ch=conv_ch, res_ch=96, taps=1, dilations=(1, 1))
    frames = synth.make_cond(rows, rows * L // synth.HOP + 2, synth.COND_DIM)
    m, q = B.wrnn_create(w, dtype, max_batch=rows), B.wrnn_subscale_net_create(nw)
    try:
        out = torch.zeros(rows * L, dtype=torch.int16, device="cuda:0")
        B.wrnn_sample_subscale_net(m, q, torch.from_numpy(frames).cuda(), 64, 64, lag, rows * L, SEED, out)
        torch.cuda.synchronize()
        assert B.wrnn_poll_status(m) == 0 and B.wrnn_subscale_net_status(q) == 0
    finally:
        B.wrnn_subscale_net_destroy(q)
        B.wrnn_destroy(m)
    got, om, net = orc.fold(out.cpu().numpy(), rows), orc.OracleModel(w, dtype), sn.SubscaleNet(nw)

    def wrong(s):
        c, f = pu._split(got[s])
        cond = frames[s][(rows * np.arange(L) + s) // synth.HOP] + net.conditioning(got, s)
        r = om.run(cond[None], L, 1, SEED, hop=1, stream0=s, c_forced=c, f_forced=f)
        return [pu.check_indices(x, y[0], r.margins[0, :, k])[1] for x, y, k in ((c, r.c_out, 0), (f, r.f_out, 1))]

    with ThreadPoolExecutor(pu.NCPU) as ex:
        assert all(n == [0, 0] for n in ex.map(wrong, sorted({0, 1, rows // 3, rows // 2, rows - 2, rows - 1})))
