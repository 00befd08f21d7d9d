"""The cluster-resident kernel of five to fourteen rows per cluster: two pipes of up to four, six and seven rows, partial last clusters,
one and several waves."""
import numpy as np
import pytest

from oracle import wrnn_oracle as orc
from paper_1802_08435_b200 import synth
from tests import parity_util as pu
from tests.test_gpu_parity import _free_run, _tol_check
from tests.test_gpu_resident_edges import _run64, _state

pytestmark = pytest.mark.gpu

SEED = synth.SEED_SAMPLING


# rows -> rows per cluster (clusters): 29 -> 5 (6, the last one 4), 43 -> 7 (7, the last one 1: a pipe without rows), 70 -> 10 (7), 78 -> 12 (7, 6),
# 85 -> 13 (7, 7), 98 -> 14 (7), 225 -> 11 (21, 5)
@pytest.mark.parametrize("rows", [29, 43, 70, 78, 85, 98, 225])
def test_rows_kernel(rows, monkeypatch):
    """Teacher-forced against the oracle; a call in pieces, down to single steps, equals one call; the checked form draws the same samples; the
    errors against 64 bits stay below those of the kernel before it (2-norms 0.92e-7 gates, 1.75e-7 state, 2.30e-7 logits)."""
    import torch
    from paper_1802_08435_b200 import binding as B
    w = synth.make_weights(896)
    cond = synth.make_cond(rows, 40, seed=3)
    kw = dict(hop=10, row_stride=3, row_offset_mul=1, stream0=5)
    m = B.wrnn_create(w, "bf16", max_batch=rows)
    try:
        r = pu.teacher_forced_parity(torch, B, m, orc.OracleModel(w, "bf16"), cond, 30, rows, SEED, threads=pu.NCPU, **kw)
        _tol_check(r, "bf16")
        whole = _free_run(torch, B, m, cond, 30, rows, SEED, **kw)
        st = _state(torch, rows)
        pieces = [_free_run(torch, B, m, cond, n, rows, SEED, step0=s, **kw, **st) for s, n in [(0, 13), (13, 1), (14, 1), (15, 15)]]
        assert np.array_equal(np.concatenate(pieces, axis=1), whole)
        # one row with a state beyond what the operand images hold: its cluster takes plain steps until it has come back; the others draw as before
        st = _state(torch, rows)
        st["h"][rows // 2, :5] = 30.0
        odd = _free_run(torch, B, m, cond, 30, rows, SEED, **kw, **st)
        per = -(-rows // (B.wrnn_launch_info(m, rows)["n_ctas"] // 16))
        far = [b for b in range(rows) if b // per != (rows // 2) // per]
        assert np.array_equal(odd[far], whole[far]) and np.isfinite(st["h"].cpu().numpy()).all()
        if rows < 200:
            rng = np.random.default_rng(1)
            T, z = 100, lambda *s: torch.zeros(s, dtype=torch.float32, device="cuda:0")
            d = (z(T, rows, 3 * 896), z(T, rows, 896), z(T, rows, 2, 256))
            sym = rng.integers(0, 256, (rows, T, 2))
            u = lambda k: torch.from_numpy(sym[:, :, k].astype(np.uint8).copy()).cuda()
            B.wrnn_step_teacher_forced(m, torch.from_numpy(cond).cuda(), T, rows, SEED, u(0), u(1), u(0), u(1), dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2])
            torch.cuda.synchronize()
            err = [((got.double() - want).norm() / want.norm()).item() for got, want in zip(d, _run64(torch, w, "bf16", cond, sym[..., None] / 127.5 - 1, False))]
            print("\n[64 bits] %d rows: gates %.2e state %.2e logits %.2e" % (rows, *err))
            assert all(e <= b for e, b in zip(err, (0.92e-7, 1.75e-7, 2.30e-7))), err
    finally:
        B.wrnn_destroy(m)
    monkeypatch.setenv("WRNN_DEBUG", "1")
    m = B.wrnn_create(w, "bf16", max_batch=rows)
    try:
        assert np.array_equal(_free_run(torch, B, m, cond, 30, rows, SEED, **kw), whole)
    finally:
        B.wrnn_destroy(m)


# last clusters of one row, whose second pipe has none: 31 -> 5 rows per cluster (7 clusters), 131 -> 10 (14), 183 -> 14 (14)
@pytest.mark.parametrize("rows", [31, 131, 183])
def test_rows_kernel_pipe_without_rows(rows):
    """A pipe without rows takes part in nothing, in calls as short as one step: these draw what one call draws."""
    import torch
    from paper_1802_08435_b200 import binding as B
    cond, n = synth.make_cond(rows, 2), 30
    m = B.wrnn_create(synth.make_weights(896), "bf16", max_batch=rows)
    try:
        per = -(-rows // (B.wrnn_launch_info(m, rows)["n_ctas"] // 16))
        assert rows % per == 1
        whole, cond_d = _free_run(torch, B, m, cond, n, rows, SEED), torch.from_numpy(cond).cuda()
        for _ in range(3):
            st, out = _state(torch, rows), torch.zeros((n, rows, 1), dtype=torch.int16, device="cuda:0")
            for i in range(n):
                B.wrnn_sample(m, cond_d, 1, rows, SEED, out[i], step0=i, **st)
            torch.cuda.synchronize()
            assert B.wrnn_poll_status(m) == 0 and np.array_equal(out.cpu().numpy()[:, :, 0].T, whole)
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("rows", [37, 98])
def test_rows_kernel_phases(rows):
    """The stamps of the first warp have names of their own, all of them are taken, and they neither change what is drawn nor exceed the call."""
    import torch
    from paper_1802_08435_b200 import binding as B
    cond, n = synth.make_cond(rows, 3), 240
    m = B.wrnn_create(synth.make_weights(896), "bf16", max_batch=rows)
    try:
        plain = _free_run(torch, B, m, cond, n, rows, SEED)
        B.wrnn_phase_profile(m, True)
        assert np.array_equal(_free_run(torch, B, m, cond, n, rows, SEED), plain)
        cycles, names = B.wrnn_phase_cycles(m), B.wrnn_phase_names(m)
        phases = ["wait_y", "hid_products", "hid_sums", "wait_background", "log_products_send", "gates_prepare", "wait_symbol", "gates"]
        assert names == [h + p for h in ("F.", "C.") for p in phases]
        print("\n[phases] %d rows, cycles per step: %s" % (rows, ", ".join("%s %.0f" % (k, c / n) for k, c in zip(names, cycles))))
        assert min(cycles) > 0 and 2000 * n < sum(cycles) < 40000 * n, cycles
    finally:
        B.wrnn_destroy(m)


@pytest.mark.parametrize("rows,big", [(43, 30.0), (78, 1e6), (98, 30.0)])
def test_rows_kernel_large_states(rows, big):
    """A row whose state is beyond what the operand images hold, in a cluster of seven, twelve and fourteen rows: its cluster takes plain steps until
    it has come back, and every row -- those beside it in either pipe, those of the other clusters -- follows the oracle in gates, states, logits, draws
    and the final state; so does a row that comes back after the first step.  (The large row itself in its first gates, within the rounding of its sums.)"""
    import torch
    from paper_1802_08435_b200 import binding as B
    n, H, dev = 24, 896, "cuda:0"
    w, cond = synth.make_weights(H), synth.make_cond(rows, 2)
    h0 = np.tanh(np.random.default_rng(5).standard_normal((rows, H))).astype(np.float32)
    odd, back = rows // 2, 1                                             # (clusters of their own)
    h0[odd, ::7] *= np.float32(big)
    h0[back, int(np.argmin(np.diag(w["R"][:H])))] = big                  # a unit that its own update gate takes back at once
    ref = orc.OracleModel(w, "bf16").run(cond, n, rows, SEED, dump=True, h=h0, threads=pu.NCPU)
    z = lambda *s: torch.zeros(s, dtype=torch.float32, device=dev)
    m = B.wrnn_create(w, "bf16", max_batch=rows)
    try:
        per = -(-rows // (B.wrnn_launch_info(m, rows)["n_ctas"] // 16))
        assert odd // per != back // per
        h, c, f = torch.from_numpy(h0).to(dev), torch.from_numpy(ref.c_out).to(dev), torch.from_numpy(ref.f_out).to(dev)
        d, co, fo = (z(n, rows, 3 * H), z(n, rows, H), z(n, rows, 2, 256)), torch.zeros_like(c), torch.zeros_like(f)
        B.wrnn_step_teacher_forced(m, torch.from_numpy(cond).to(dev), n, rows, SEED, c, f, co, fo, dbg_gates=d[0], dbg_h=d[1], dbg_logits=d[2], h=h)
        torch.cuda.synchronize()
        assert B.wrnn_poll_status(m) == 0, B.wrnn_last_error(m)
    finally:
        B.wrnn_destroy(m)
    got = [x.cpu().numpy().reshape(n, rows, -1) for x in d] + [h.cpu().numpy()[None]]
    want = [np.asarray(x).reshape(n, rows, -1) for x in (ref.gates, ref.hs, ref.logits)] + [np.asarray(ref.h)[None]]
    rest = [b for b in range(rows) if b != odd]
    for g, r in zip(got, want):
        assert np.isfinite(g).all() and pu.rel_err(g[:, rest], r[:, rest]) < pu.TOL["bf16"]
    for x, y, k in ((co, ref.c_out, 0), (fo, ref.f_out, 1)):
        assert pu.check_indices(x.cpu().numpy()[rest], y[rest], ref.margins[rest][:, :, k])[1] == 0
    # sums of fp32 terms, (terms) x 2^-24 x sum |term|; gates of slope one at most
    bound = H * 2.0 ** -24 * (np.abs(w["R"]).astype(np.float64) @ np.abs(h0[odd]).astype(np.float64)).max()
    assert np.abs(got[0][0, odd] - want[0][0, odd]).max() < pu.TOL["bf16"] + bound


@pytest.mark.parametrize("rows", [78, 98])
def test_rows_kernel_lost_word(rows):
    """The wider forms (pipes of six and seven rows) when a CTA of every cluster withholds the state it publishes at one step: the waits that depend on
    it run out, the call reports where and returns, and the model works again."""
    import re
    import torch
    from paper_1802_08435_b200 import binding as B
    cond, n, at = synth.make_cond(rows, 2), 60, 23
    m = B.wrnn_create(synth.make_weights(896), "bf16", max_batch=rows)
    try:
        ref = _free_run(torch, B, m, cond, n, rows, SEED)
        n_ctas = B.wrnn_launch_info(m, rows)["n_ctas"]
        B.wrnn_selftest_lost_word(m, 4_000_000, n_ctas // 2, at)
        out = torch.zeros((rows, n), dtype=torch.int16, device="cuda:0")
        B.wrnn_sample(m, torch.from_numpy(cond).cuda(), n, rows, SEED, out)
        torch.cuda.synchronize()
        assert B.wrnn_poll_status(m) == B.WRNN_ERR_TIMEOUT
        cta, step, _ = (int(x) for x in re.search(r"at cta (-?\d+), step (-?\d+), phase (-?\d+)", B.wrnn_last_error(m)).groups())
        assert 0 <= cta < n_ctas and at <= step <= at + 1, B.wrnn_last_error(m)
        B.wrnn_selftest_lost_word(m, 0, -1, -1)
        assert np.array_equal(_free_run(torch, B, m, cond, n, rows, SEED), ref)
    finally:
        B.wrnn_destroy(m)


def test_rows_kernel_staggered():
    """Dependent rows on the staggered schedule with up to forty of them under way at once: every draw against the oracle conditioned on the device's
    samples."""
    import torch
    from paper_1802_08435_b200 import binding as B
    from tests.test_gpu_subscale_dep import _case, _gpu_run
    rows, L, F, chunk = 40, 360, 4, 4
    w, V, b, frames = _case(896, rows, L, F, scale=1.0)
    m = B.wrnn_create(w, "bf16", max_batch=rows)
    try:
        got = orc.fold(_gpu_run(torch, B, m, frames, V, b, F, chunk, 8, rows, L), rows)
        want, _, mg = orc.subscale_dependent_run(orc.OracleModel(w, "bf16"), frames, V, b, rows, L, synth.HOP, SEED, forced=got, teacher=True)
        for g, r, k in zip(pu._split(got), pu._split(want), (0, 1)):
            assert pu.check_indices(g, r, mg[:, :, k])[1] == 0
    finally:
        B.wrnn_destroy(m)
