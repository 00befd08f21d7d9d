"""Calls at the edges of what the resident kernels take: short calls, caller-supplied states, many models at once."""
import numpy as np
import pytest

from oracle import wrnn_oracle as orc
from paper_1802_08435_b200 import synth
from tests import parity_util as pu
from tests.test_gpu_parity import _free_run

pytestmark = pytest.mark.gpu

SEED = synth.SEED_SAMPLING


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1802_08435_b200 import binding as B
    assert torch.cuda.is_available()
    return torch, B


def _state(torch, batch, H=896):
    return dict(h=torch.zeros((batch, H), dtype=torch.float32, device="cuda:0"),
                c_prev=torch.full((batch,), 128, dtype=torch.uint8, device="cuda:0"),
                f_prev=torch.zeros((batch,), dtype=torch.uint8, device="cuda:0"))


@pytest.mark.parametrize("dtype,batch", [("bf16", 1), ("bf16", 7), ("bf16", 27), ("bf16", 56), ("f32", 1), ("f32", 27)])
def test_calls_of_one_step_equal_one_call(env, dtype, batch):
    """Every call multiplies R by the state that it is given before the CTAs of a cluster exchange their first new one, and a CTA that
    is ahead must not store that over the state that another one still reads.  Calls of one step are nothing but this: all forms of
    the cluster-resident kernels (one, up to four, up to eight rows per cluster), against one call."""
    torch, B = env
    n = 60
    cond = synth.make_cond(batch, 2)
    m = B.wrnn_create(synth.make_weights(896), dtype, max_batch=batch)
    try:
        whole = _free_run(torch, B, m, cond, n, batch, SEED)
        for _ in range(3):
            st = _state(torch, batch)
            cond_d = torch.from_numpy(cond).cuda()
            out = torch.zeros((n, batch, 1), dtype=torch.int16, device="cuda:0")
            for i in range(n):
                B.wrnn_sample(m, cond_d, 1, batch, SEED, out[i], step0=i, **st)
            torch.cuda.synchronize()
            assert B.wrnn_poll_status(m) == 0
            assert np.array_equal(out.cpu().numpy()[:, :, 0].T, whole)
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("case", ["sparse", "f32", "batched"])
def test_a_smaller_model_leaves_a_larger_one_its_shared_memory(env, monkeypatch, case):
    """What a kernel may ask for is set per function, not per model: creating a model that needs less must not refuse the launches of
    one that is alive and needs more."""
    torch, B = env
    if case == "sparse":
        # four clusters, whose shared memory grows with the kept blocks
        monkeypatch.setenv("WRNN_SPARSE_CLUSTERS", "4")
        mk = lambda sparsity: B.wrnn_create(synth.make_weights(2048), "bf16", synth.make_block_masks(2048, sparsity), kernel=B.WRNN_KERNEL_SPARSE)
        sizes = (0.88, 0.96)
    else:
        kern = B.WRNN_KERNEL_BATCHED if case == "batched" else B.WRNN_KERNEL_RESIDENT
        dtype, batch = ("f32", 1) if case == "f32" else ("bf16", 2 if case == "batched" else 1)
        mk = lambda H: B.wrnn_create(synth.make_weights(H), dtype, max_batch=batch, kernel=kern)
        sizes = {"f32": (832, 192), "batched": (1024, 128)}[case]
    rows = 2 if case == "batched" else 1
    cond = synth.make_cond(rows, 2)
    models = [mk(s) for s in sizes]
    try:
        infos = [B.wrnn_launch_info(m, rows) for m in models]
        assert infos[0]["kernel"] == infos[1]["kernel"] and infos[0]["smem_bytes"] > infos[1]["smem_bytes"], infos
        for m in models:
            _free_run(torch, B, m, cond, 20, rows, SEED)
    finally:
        for m in models:
            B.wrnn_destroy(m)


@pytest.mark.parametrize("case", ["bf16", "f32", "fused", "sparse", "sparse16x1"])
@pytest.mark.parametrize("big", [1.5, 30.0, 1e6, 1e20])
def test_states_beyond_one(env, case, big):
    """A caller may hand over any state.  A row whose state is far outside (-1, 1) follows the oracle like any other, while it is
    large and once it has come back, and leaves the rows beside it alone: they draw what they draw without it."""
    torch, B = env
    n, hop = 24, 120
    rng = np.random.default_rng(5)
    dev = "cuda:0"
    sparse = case.startswith("sparse")
    H, rows = (2048 if sparse else 896), (1 if sparse or case == "fused" else 6)
    dtype = "f32" if case == "f32" else "bf16"
    masks, block = None, (16, 1) if case == "sparse16x1" else (4, 4)
    if case == "fused":
        w = synth.make_weights(H, n_inputs=12, n_logits=64)
    else:
        w = synth.make_weights(H)
    if sparse:
        masks = synth.make_block_masks(H, 0.96, block=block)
        w = synth.rescale_kept(w, masks)
    h0 = np.tanh(rng.standard_normal((rows, H))).astype(np.float32)
    # one unit that its own update gate takes back at once, in every case; beside it a row of which units stay large
    R = w["R"][:H, :H] if masks is None else w["R"][:H, :H] * np.repeat(np.repeat(masks["R"][:H // block[0]], block[0], 0), block[1], 1)
    odd, k_back = rows // 2, int(np.argmin(np.diag(R)))
    h0[max(odd - 1, 0), k_back] = big
    if rows > 1:
        h0[odd, ::7] *= np.float32(big)
    cond = synth.make_cond(rows, 2)
    m = B.wrnn_create(w, dtype, masks, max_batch=28 if rows > 1 else 1, block=block, variant=1 if case == "fused" else 0)
    tol = pu.TOL[dtype]

    def forced(sel):
        """gates, states and logits of a call that is given the states of the rows `sel`, against the oracle's"""
        k = len(sel)
        h = torch.from_numpy(h0[sel]).to(dev)
        z = lambda *s: torch.zeros(s, dtype=torch.float32, device=dev)
        if case == "fused":
            ref = orc.Fs2OracleModel(w, "bf16").run(cond[0], n, seed=SEED, hop=hop, dump=True, h=h0[0])
            u16 = lambda a: torch.from_numpy(a.astype(np.uint16).view(np.int16).copy()).to(dev)
            d = (z(n, 3 * H), z(n, H), z(n, 2, 64))
            a, b = u16(ref.a_out), u16(ref.b_out)
            B.wrnn_fs2_step_teacher_forced(m, torch.from_numpy(cond).to(dev), n, SEED, a, b, torch.zeros_like(a), torch.zeros_like(b),
                                           dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2], hop=hop, h=h[0])
        else:
            ref = orc.OracleModel(w, dtype, masks, block).run(cond[sel], n, k, SEED, stream0=0, dump=True, h=h0[sel], threads=pu.NCPU)
            c, f = torch.from_numpy(ref.c_out).to(dev), torch.from_numpy(ref.f_out).to(dev)
            d = (z(n, k, 3 * H), z(n, k, H), z(n, k, 2, 256))
            B.wrnn_step_teacher_forced(m, torch.from_numpy(cond[sel]).to(dev), n, k, SEED, c, f, torch.zeros_like(c), torch.zeros_like(f),
                                       dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2], h=h)
        torch.cuda.synchronize()
        assert B.wrnn_poll_status(m) == 0, B.wrnn_last_error(m)
        got = [x.cpu().numpy().reshape(n, k, -1) for x in d] + [h.cpu().numpy().reshape(1, k, -1)]
        want = [np.asarray(x).reshape(n, k, -1) for x in (ref.gates, ref.hs, ref.logits)] + [np.asarray(ref.h).reshape(1, k, -1)]
        # The row that stays large: its sums have terms of up to `big` and are exact to (terms) x 2^-24 x sum |term| in fp32, in
        # whatever kernel, which near a zero of the sum is no longer small.  Its first gates (of slope one at most) lie within that.
        rest = [i for i, r in enumerate(sel) if rows == 1 or r != odd]
        for g, r in zip(got, want):
            assert np.isfinite(g).all() and pu.rel_err(g[:, rest], r[:, rest]) < tol
        if rows > 1:
            bound = H * 2.0 ** -24 * (np.abs(w["R"]).astype(np.float64) @ np.abs(h0[odd]).astype(np.float64)).max()
            assert np.abs(got[0][0, odd] - want[0][0, odd]).max() < tol + bound

    try:
        if rows == 1:
            forced([0])
        else:
            forced(list(range(rows)))                                    # one row per cluster
            cond_28 = np.concatenate([cond, synth.make_cond(22, 2, seed=9)])
            h_28 = np.concatenate([h0, np.tanh(rng.standard_normal((22, H))).astype(np.float32)])
            outs = []
            for scale in (1.0, 0.0):                                     # four rows per cluster: with the large state, without it
                h = h_28.copy()
                h[[odd - 1, odd]] *= scale
                st = dict(_state(torch, 28), h=torch.from_numpy(h).to(dev))
                outs.append(_free_run(torch, B, m, cond_28, n, 28, SEED, **st))
                assert np.isfinite(st["h"].cpu().numpy()).all()
                outs.append(st["h"].cpu().numpy())
            others = [r for r in range(28) if r not in (odd - 1, odd)]
            assert np.array_equal(outs[0][others], outs[2][others])
            assert np.abs(outs[1][others] - outs[3][others]).max() < 1e-5
    finally:
        B.wrnn_destroy(m)


def _run64(torch, w, dtype, cond, x, fused):
    """gates, states and logits of a teacher-forced call in 64 bits.  x [rows][steps][2][1 or 4]: the coarse and fine symbols as
    the network sees them."""
    dev = "cuda:0"
    rows, T, _, nx = x.shape
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    cast = (lambda a: t(a).bfloat16().double()) if dtype == "bf16" else (lambda a: t(a).double())
    W = {k: cast(w[k]) for k in ("R", "I", "W_cond", "O1", "O2", "O3", "O4")}
    b = {k: t(w[k]).double() for k in ("b_gate", "b1", "b2", "b3", "b4")}
    H = W["R"].shape[1]
    half = H // 2
    for g in range(3):
        W["I"][g * H:g * H + half, 2 * nx:] = 0                         # the coarse half does not see this step's coarse symbol
    off = t(cond).double() @ W["W_cond"].T + b["b_gate"]
    first = [np.array([8, 0, 0, 0]) / 7.5 - 1] * 2 if fused else [np.array([128 / 127.5 - 1]), np.array([-1.0])]
    prev = [t(np.broadcast_to(f, (rows, nx)).copy()).double() for f in first]
    X, h = t(x).double(), torch.zeros(rows, H, dtype=torch.double, device=dev)
    gates, hs, logits = [], [], []
    for s in range(T):
        a, i = h @ W["R"].T, torch.cat([*prev, X[:, s, 0]], 1) @ W["I"].T + off[:, s // 120]
        u, r = torch.sigmoid(a[:, :H] + i[:, :H]), torch.sigmoid(a[:, H:2 * H] + i[:, H:2 * H])
        e = torch.tanh(r * a[:, 2 * H:] + i[:, 2 * H:])
        h = u * h + (1 - u) * e
        gates.append(torch.cat([u, r, e], 1))
        hs.append(h)
        logits.append(torch.stack([torch.relu(h[:, :half] @ W["O1"].T + b["b1"]) @ W["O2"].T + b["b2"],
                                   torch.relu(h[:, half:] @ W["O3"].T + b["b3"]) @ W["O4"].T + b["b4"]], 1))
        prev = [X[:, s, 0], X[:, s, 1]]
    return [torch.stack(v) for v in (gates, hs, logits)]


@pytest.mark.parametrize("dtype,rows", [("bf16", 1), ("bf16", 7), ("f32", 1), ("f32", 7), ("f32", 8), ("fused", 1)])
def test_error_against_64_bits(env, dtype, rows):
    """The cluster-resident kernel multiplies on the tensor cores, in two parts of 11 bits and with sums that are cut off; this must
    not cost precision.  The bounds are the 2-norms of the errors of the kernels before it, which multiplied exact operands (bf16,
    one row: 1.03e-7 gates, 1.92e-7 state, 2.04e-7 logits; fused 1.05, 1.96, 2.23; fp32 1.03, 1.95, 2.12, several rows 0.82, 1.66, 1.96)."""
    torch, B = env
    T, H, dev, fused = 200, 896, "cuda:0", dtype == "fused"
    bound = (0.83e-7, 1.7e-7, 2.0e-7) if dtype == "f32" and rows > 1 else (1.05e-7, 1.96e-7, 2.12e-7)
    for seed in (1, 2):
        rng = np.random.default_rng(seed)
        w = synth.make_weights(H, seed_w=seed, seed_b=seed + 1, **(dict(n_inputs=12, n_logits=64) if fused else {}))
        cond = synth.make_cond(rows, 2, seed=seed + 3)
        z = lambda *s: torch.zeros(s, dtype=torch.float32, device=dev)
        d = (z(T, rows, 3 * H), z(T, rows, H), z(T, rows, 2, 64 if fused else 256))
        sym = rng.integers(0, 65536 if fused else 256, (rows, T, 2))
        u = lambda k: torch.from_numpy(sym[:, :, k].astype(np.uint16 if fused else np.uint8).view(np.int16 if fused else np.uint8).copy()).to(dev)
        m = B.wrnn_create(w, "bf16" if fused else dtype, max_batch=rows, variant=1 if fused else 0)
        try:
            if fused:
                x = np.stack([(sym >> s) & 15 for s in (12, 8, 4, 0)], -1) / 7.5 - 1
                B.wrnn_fs2_step_teacher_forced(m, torch.from_numpy(cond).to(dev), T, SEED, u(0)[0], u(1)[0], u(0)[0].clone(), u(1)[0].clone(),
                                               dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2])
            else:
                x = sym[..., None] / 127.5 - 1
                B.wrnn_step_teacher_forced(m, torch.from_numpy(cond).to(dev), T, rows, SEED, u(0), u(1), u(0).clone(), u(1).clone(),
                                           dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2])
            torch.cuda.synchronize()
            assert B.wrnn_poll_status(m) == 0
        finally:
            B.wrnn_destroy(m)
        err = [((got.double() - want).norm() / want.norm()).item() for got, want in zip(d, _run64(torch, w, "bf16" if fused else dtype, cond, x, fused))]
        print("\n[64 bits] %s, %d rows: gates %.2e state %.2e logits %.2e" % (dtype, rows, *err))
        assert all(e <= b for e, b in zip(err, bound)), (err, bound)


@pytest.mark.parametrize("rows", [1, 16, 37])
def test_short_wait_limits_leave_copies_their_time(env, rows):
    """A wait covers the copies that bring a CTA's own weights on chip: a limit below what these take, which a caller may ask for, does not let
    the CTA leave before they have landed.  Nothing is withheld here, so the call ends as any other."""
    torch, B = env
    cond = synth.make_cond(rows, 2)
    m = B.wrnn_create(synth.make_weights(896), "bf16", max_batch=rows)
    try:
        want = _free_run(torch, B, m, cond, 20, rows, SEED)
        for limit in (1, 1000):
            B.wrnn_selftest_lost_word(m, limit, -1, -1)
            assert np.array_equal(_free_run(torch, B, m, cond, 20, rows, SEED), want) and B.wrnn_poll_status(m) == 0
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("case,rows", [("bf16", 1), ("bf16", 16), ("bf16", 37), ("f32", 1), ("fused", 1)])
def test_captured_calls(env, case, rows):
    """A call in a graph -- a lone cluster is launched beside the projection of its frames there too -- and pieces that hand the state on from one
    call to the next: every replay draws what the calls draw."""
    torch, B = env
    n, fused, dev = 30, case == "fused", "cuda:0"
    w = synth.make_weights(896, **(dict(n_inputs=12, n_logits=64) if fused else {}))
    cond = torch.from_numpy(synth.make_cond(rows, 2)).cuda()
    m = B.wrnn_create(w, "f32" if case == "f32" else "bf16", max_batch=rows, variant=1 if fused else 0)
    out = torch.zeros((3, 2 if fused else rows, n), dtype=torch.int16, device=dev)
    st = {} if fused else _state(torch, rows)
    h0 = torch.zeros((rows, 896), device=dev)

    def calls():
        if fused:
            h0.zero_()
            for i in range(3):
                B.wrnn_fs2_sample(m, cond, n, SEED, out[i], h=h0, step0=n * i)
            return
        st["h"].zero_(), st["c_prev"].fill_(128), st["f_prev"].zero_()
        for i in range(3):
            B.wrnn_sample(m, cond, n, rows, SEED, out[i], step0=n * i, **st)

    try:
        calls()
        torch.cuda.synchronize()
        want = out.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            calls()
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert B.wrnn_poll_status(m) == 0 and torch.equal(out, want)
        del graph
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("case,rows", [("bf16", 1), ("bf16", 6), ("bf16", 30), ("f32", 3), ("fused", 1)])
def test_states_at_any_address(env, case, rows):
    """A caller's state is an array of floats: one that starts between two 16-byte boundaries gives what an aligned one gives, also where it is
    so large that the cluster takes plain steps."""
    torch, B = env
    n, fused = 20, case == "fused"
    w = synth.make_weights(896, **(dict(n_inputs=12, n_logits=64) if fused else {}))
    cond = torch.from_numpy(synth.make_cond(rows, 2)).cuda()
    m = B.wrnn_create(w, "f32" if case == "f32" else "bf16", max_batch=rows, variant=1 if fused else 0)
    h0 = torch.from_numpy(np.random.default_rng(3).uniform(-0.9, 0.9, (rows, 896)).astype(np.float32)).cuda()
    try:
        for big in (0.5, 30.0):
            h0[rows // 2, 7] = big
            got = []
            for shift in (0, 1, 3):
                h = torch.zeros(rows * 896 + 4, device="cuda:0")[shift:shift + rows * 896].view(rows, 896)
                assert h.data_ptr() % 16 == 4 * shift
                h.copy_(h0)
                out = torch.zeros((2 if fused else rows, n), dtype=torch.int16, device="cuda:0")
                if fused:
                    B.wrnn_fs2_sample(m, cond, n, SEED, out, h=h)
                else:
                    B.wrnn_sample(m, cond, n, rows, SEED, out, h=h)
                torch.cuda.synchronize()
                assert B.wrnn_poll_status(m) == 0
                got.append((out.cpu(), h.cpu()))
            assert all(torch.equal(a, b) for g in got[1:] for a, b in zip(g, got[0]))
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("H,rows,kernel", [(128, 11, "BCLUSTER"), (128, 11, "BATCHED"), (896, 3, "AUTO"), (896, 30, "AUTO"), (64, 2, "GENERIC")])
def test_dumps_at_any_address(env, H, rows, kernel):
    """Gates, states and logits are written as floats, wherever the caller's arrays start."""
    torch, B = env
    n, dev = 12, "cuda:0"
    cond = torch.from_numpy(synth.make_cond(rows, 2)).cuda()
    forced = torch.from_numpy(np.random.default_rng(4).integers(0, 256, (2, rows, n)).astype(np.uint8)).cuda()
    m = B.wrnn_create(synth.make_weights(H), "bf16", max_batch=rows, kernel=getattr(B, "WRNN_KERNEL_" + kernel))
    try:
        got = []
        for shift in (0, 1):
            d = [torch.zeros(n * rows * k + 4, device=dev)[shift:shift + n * rows * k].view(n, rows, k) for k in (3 * H, H, 512)]
            c, f = torch.zeros_like(forced[0]), torch.zeros_like(forced[1])
            B.wrnn_step_teacher_forced(m, cond, n, rows, SEED, forced[0], forced[1], c, f, dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2].view(n, rows, 2, 256))
            torch.cuda.synchronize()
            assert B.wrnn_poll_status(m) == 0
            got.append([x.cpu() for x in (*d, c, f)])
        assert all(torch.equal(a, b) for a, b in zip(*got)) and got[0][2].abs().min() > 0
    finally:
        B.wrnn_destroy(m)


def test_first_subscale_call_costs_little_more_than_the_next(env):
    """A staggered schedule starts with one active row and adds one per lag: its workspaces are made for the largest call at once, not
    regrown (with a device synchronisation each time) on the way.  Best of three fresh models, room for the kernels' first loads."""
    import time
    torch, B = env
    rows, L = 16, 3200
    frames = torch.from_numpy(synth.make_cond(rows, rows * L // 120 + 1)).cuda()
    out = torch.zeros(rows * L, dtype=torch.int16, device="cuda:0")
    first, again = [], []
    for _ in range(4):
        m = B.wrnn_create(synth.make_weights(896), "bf16", max_batch=rows)
        net = B.wrnn_subscale_net_create(synth.make_subscale_net(rows))
        try:
            for times in (first, again):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                B.wrnn_sample_subscale_net(m, net, frames, 128, 128, 256, rows * L, SEED, out)
                torch.cuda.synchronize()
                times.append(time.perf_counter() - t0)
        finally:
            B.wrnn_subscale_net_destroy(net)
            B.wrnn_destroy(m)
    print("\n[first call] %s ms, repeated %s ms" % tuple(["%.1f" % (1e3 * t) for t in x] for x in (first, again)))
    assert min(first[1:]) < 1.5 * min(again)


def test_creating_an_fp32_model_costs_little_more_than_a_bf16_one(env):
    """Packing splits every fp32 weight in two and lays it out twice, on several host threads.  Best of six, fp32 against bf16 (20 and
    18 ms; 55 and 45 and more on one thread, which took 1.7 times as long for fp32 on an idle host)."""
    import time
    torch, B = env
    w, best = synth.make_weights(896), {}
    for _ in range(6):
        for dtype in ("f32", "bf16"):
            t0 = time.perf_counter()
            m = B.wrnn_create(w, dtype)
            torch.cuda.synchronize()
            best[dtype] = min(best.get(dtype, 1e9), time.perf_counter() - t0)
            B.wrnn_destroy(m)
    print("\n[create] fp32 %.1f ms, bf16 %.1f ms" % (1e3 * best["f32"], 1e3 * best["bf16"]))
    assert best["f32"] < 1.5 * best["bf16"]


@pytest.mark.parametrize("dtype,H", [("bf16", 896), ("f32", 896), ("bf16", 2048)])
def test_draws_from_logits_that_are_not_finite(env, dtype, H):
    """Symbols that a bias of minus infinity forbids are never drawn; where a logit is not a number no running sum exceeds the
    threshold, and the last symbol is drawn, as in the oracle."""
    torch, B = env
    masks = synth.make_block_masks(H, 0.96) if H == 2048 else None
    w = synth.make_weights(H)
    cond = synth.make_cond(1, 2)
    for case in ("forbid", "nan", "nan_first"):
        w["b2"] = np.zeros(256, np.float32)
        if case == "forbid":
            w["b2"][40:200] = -np.inf
        else:
            w["b2"][0 if case == "nan_first" else 77] = np.nan
        m = B.wrnn_create(w, dtype, masks)
        try:
            out = _free_run(torch, B, m, cond, 60, 1, SEED)
            coarse = (out[0].astype(np.int32) + 32768) >> 8
            if case == "forbid":
                ref = orc.OracleModel(w, dtype, masks).run(cond, 60, 1, SEED, dump=True)
                div = pu.first_divergence(out, ref.out)
                assert ((coarse < 40) | (coarse >= 200)).all() and (div < 0 or ref.margins[0, div].min() < pu.MARGIN)
            else:
                assert (coarse == 255).all(), coarse
        finally:
            B.wrnn_destroy(m)


@pytest.mark.parametrize("dtype,H", [("bf16", 896), ("f32", 896), ("bf16", 2048)])
@pytest.mark.parametrize("case", ["unit_off", "unit_off_inf", "tiny_head", "tiny_hidden", "tiny_recurrent", "unit_on"])
def test_scales_of_unusual_weights(env, dtype, H, case):
    """The fp16 operands are scaled by powers of two taken from the weights and biases: units that a large negative bias switches off
    (finite or not) must not take the scale of the others with them, a large positive one may, and matrices whose scale would not be a
    number keep a finite one."""
    torch, B = env
    masks = synth.make_block_masks(H, 0.96) if H == 2048 else None
    w = synth.make_weights(H)
    if case.startswith("unit_off"):
        w["b1"][5], w["b3"][-3] = (-np.inf, -np.inf) if case.endswith("inf") else (-1e30, -3e25)
    elif case == "unit_on":
        w["b1"][5] = 1e5
        w["O2"][:, 5] = 0                                               # large, and read by nobody
    else:
        for k in {"tiny_head": ("O2", "O4"), "tiny_hidden": ("O1", "b1", "O3", "b3"), "tiny_recurrent": ("R",)}[case]:
            w[k] = w[k] * np.float32(1e-35)
    cond = synth.make_cond(1, 2)
    om = orc.OracleModel(w, dtype, masks)
    m = B.wrnn_create(w, dtype, masks)
    try:
        r = pu.teacher_forced_parity(torch, B, m, om, cond, 60, 1, SEED)
        tol = pu.TOL[dtype]
        assert r["idx_bad"] == 0 and r["gates_err"] < tol and r["h_err"] < tol and r["logits_err"] < tol, {k: v for k, v in r.items() if k != "oracle"}
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("dtype,rows,clusters", [("bf16", 1, 1), ("bf16", 4, 4), ("bf16", 7, 7), ("bf16", 8, 4), ("bf16", 56, 7), ("bf16", 57, 12), ("bf16", 224, 28),
                                                 ("f32", 1, 1), ("f32", 8, 4), ("f32", 14, 7), ("f32", 15, 8)])
def test_cluster_resident_launches_only_clusters_with_rows(env, dtype, rows, clusters):
    """A cluster takes 16 SMs whether it has rows or not, and a grid is done when its last cluster is: none without rows."""
    torch, B = env
    m = B.wrnn_create(synth.make_weights(896), dtype, max_batch=rows)
    try:
        info = B.wrnn_launch_info(m, rows)
        assert info["kernel"] == B.WRNN_KERNEL_RESIDENT and info["n_ctas"] == 16 * clusters, info
        assert _free_run(torch, B, m, synth.make_cond(rows, 2), 5, rows, SEED).shape == (rows, 5)
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("dtype,most", [("bf16", 16), ("f32", 1)])
def test_resident_by_name_refuses_more_rows_than_it_says(env, dtype, most):
    torch, B = env
    m = B.wrnn_create(synth.make_weights(896), dtype, max_batch=32, kernel=B.WRNN_KERNEL_RESIDENT)
    try:
        assert _free_run(torch, B, m, synth.make_cond(most, 2), 5, most, SEED).shape == (most, 5)
        with pytest.raises(B.WrnnError):
            _free_run(torch, B, m, synth.make_cond(most + 1, 2), 5, most + 1, SEED)
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("H,rows,kernel", [(896, 224, "RESIDENT"), (896, 225, "RESIDENT"), (896, 336, "RESIDENT"), (896, 340, "BATCHED"), (1024, 224, "BCLUSTER"), (1024, 230, "BATCHED")])
def test_large_batches_run_on_the_tensor_core_kernels(env, H, rows, kernel):
    """The lines of the dispatch for many rows of a dense bf16 model: waves of the cluster-resident kernel of many rows, for other H the
    cluster-partitioned kernel, and the grid-phased one where the rows do not fit the clusters.  A few rows against the oracle."""
    torch, B = env
    w = synth.make_weights(H)
    cond = synth.make_cond(rows, 4)
    m = B.wrnn_create(w, "bf16", max_batch=rows)
    try:
        assert B.wrnn_launch_info(m, rows)["kernel"] == getattr(B, "WRNN_KERNEL_" + kernel)
        out = _free_run(torch, B, m, cond, 20, rows, SEED, row_offset_mul=1)
        chk = pu.oracle_on_gpu_stream(orc.OracleModel(w, "bf16"), cond, [0, rows // 2, rows - 1], out, SEED, row_offset_mul=1)
        assert chk["idx_bad"] == 0, chk
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("rows", [225, 256, 336])
def test_cluster_partitioned_kernel_at_many_rows(env, rows):
    """The cluster-partitioned tcgen05 kernel by name, at H = 896 and as many rows as its clusters take (several lane quadrants, ragged and full):
    rows on both sides of the cluster boundaries, every draw and the final state against the oracle forced on the device's samples."""
    torch, B = env
    w, cond = synth.make_weights(896), synth.make_cond(rows, 4)
    m = B.wrnn_create(w, "bf16", max_batch=rows, kernel=B.WRNN_KERNEL_BCLUSTER)
    try:
        info = B.wrnn_launch_info(m, rows)
        assert info["kernel"] == B.WRNN_KERNEL_BCLUSTER
        st = _state(torch, rows)
        out = _free_run(torch, B, m, cond, 40, rows, SEED, row_offset_mul=1, **st)
        per = -(-rows // (info["n_ctas"] // 16))
        some = sorted({0, per - 1, per, 2 * per, rows // 2, rows - per, rows - 1})
        chk = pu.oracle_on_gpu_stream(orc.OracleModel(w, "bf16"), cond, some, out, SEED, row_offset_mul=1, h_final=st["h"].cpu().numpy())
        assert chk["idx_bad"] == 0 and chk["h_final_err"] < pu.TOL["bf16"], chk
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("case,region", [("bf16", 6), ("rows4", 6), ("rows8", 6), ("f32", 6), ("f32x2", 6), ("fused", 6), ("sparse", 4), ("sparse16x1", 4)])
def test_checked_form_of_the_default_kernels(env, monkeypatch, case, region):
    """Models created under WRNN_DEBUG=1 run the default kernels with guards around every writable region of shared memory, their
    carve-up compared with the launch and every store into a peer range-checked: the same samples, a clean status, and one write past the
    end of a region (into its guard) reported as such."""
    torch, B = env
    rows = {"rows4": 22, "rows8": 50, "f32x2": 13}.get(case, 1)
    masks, block = None, (16, 1) if case == "sparse16x1" else (4, 4)
    if case.startswith("sparse"):
        masks = synth.make_block_masks(2048, 0.96, block=block)
    w = synth.make_weights(2048 if masks else 896, **(dict(n_inputs=12, n_logits=64) if case == "fused" else {}))
    cond = synth.make_cond(rows, 2)

    def run(m):
        if case != "fused":
            out = torch.zeros((rows, 40), dtype=torch.int16, device="cuda:0")
            B.wrnn_sample(m, torch.from_numpy(cond).cuda(), 40, rows, SEED, out)
        else:
            out = torch.zeros((2, 40), dtype=torch.int16, device="cuda:0")
            B.wrnn_fs2_sample(m, torch.from_numpy(cond).cuda(), 40, SEED, out)
        torch.cuda.synchronize()
        return out.cpu().numpy(), B.wrnn_poll_status(m)

    outs = []
    for checked in (False, True):
        if checked:
            monkeypatch.setenv("WRNN_DEBUG", "1")
        m = B.wrnn_create(w, "f32" if case.startswith("f32") else "bf16", masks, max_batch=rows, block=block, variant=1 if case == "fused" else 0)
        try:
            out, status = run(m)
            assert status == 0, B.wrnn_last_error(m)
            outs.append(out)
            if checked:
                monkeypatch.setenv("WRNN_DEBUG_POKE", "1")
                assert run(m)[1] == B.WRNN_ERR_CHECK
                assert "region %d" % region in B.wrnn_last_error(m) and "cta 3" in B.wrnn_last_error(m), B.wrnn_last_error(m)
        finally:
            B.wrnn_destroy(m)
    assert np.array_equal(*outs)


@pytest.mark.parametrize("H,dtype,rows,kernel", [(896, "bf16", 1, "AUTO"), (896, "bf16", 32, "AUTO"), (896, "f32", 2, "AUTO"), (128, "bf16", 11, "BATCHED"), (128, "bf16", 11, "BCLUSTER"),
                                                 (64, "bf16", 3, "GENERIC")])
def test_a_new_model_is_whole_on_any_stream(env, H, dtype, rows, kernel):
    """Creation returns when the weights and cleared buffers are there: the first call, on a stream that does not block with the default
    stream, draws what a later one draws."""
    torch, B = env
    w, cond, side = synth.make_weights(H), torch.from_numpy(synth.make_cond(rows, 2)).cuda(), torch.cuda.Stream()
    for _ in range(3):
        outs = [torch.zeros((rows, 20), dtype=torch.int16, device="cuda:0") for _ in range(2)]
        torch.cuda.synchronize()
        m = B.wrnn_create(w, dtype, max_batch=rows, kernel=getattr(B, "WRNN_KERNEL_" + kernel))
        try:
            for out in outs:
                B.wrnn_sample(m, cond, 20, rows, SEED, out, stream=side)
                side.synchronize()
            assert B.wrnn_poll_status(m) == 0 and torch.equal(*outs)
        finally:
            B.wrnn_destroy(m)
