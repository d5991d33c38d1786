"""GPU parity of the backward pass: ``rodimus_ddts_bwd`` through the C ABI against the fp64 adjoint
recurrence of the oracle on the same seeded inputs.  Bar, per gradient tensor:
max|err|/max|ref| <= 2e-2 (bf16 tokens: tf32 contractions, fp32 accumulation, bf16 outputs) and
<= 1e-4 (fp32 build: split-tf32 contractions at fp32 accuracy)."""
import numpy as np
import pytest

import paper_2410_06577_b200 as rd
from paper_2410_06577_b200 import workloads as wl
from oracle import ddts_oracle as orc
from tests._util import TOL_BF16, TOL_F32, dev, host, prefill_to_device, rel_err

pytestmark = pytest.mark.gpu

PAIRS = (("d_q", "dq"), ("d_k", "dk"), ("d_gate_x", "dx"), ("d_temp_y", "dy"), ("d_v", "dv"))


def _run_bwd(p, d_o, d_sT, ingate, scale, host_cu=True, want_d_s0=True):
    """Calls the library with NaN-filled outputs (an element the kernels never store stays NaN)."""
    import torch
    d = prefill_to_device(p)
    B, H, T, dk = d["q"].shape
    dv = d["v"].shape[-1]
    nseq = B if d["cu"] is None else d["cu"].numel() - 1
    g_o = dev(d_o, p.dtype)
    g_s = None if d_sT is None else torch.from_numpy(d_sT).cuda()
    out = {n: torch.full_like(d["q"], float("nan")) for n in ("d_q", "d_k", "d_gate_x", "d_temp_y")}
    out["d_v"] = torch.full_like(d["v"], float("nan"))
    out["d_s0"] = (torch.full((nseq, H, dk, dv), float("nan"), dtype=torch.float32, device="cuda")
                   if want_d_s0 else None)
    prm = rd.bwd_params(d["q"], d["k"], d["x"], d["y"], d["v"], g_o, out["d_q"], out["d_k"],
                        out["d_gate_x"], out["d_temp_y"], out["d_v"], d["s0"], g_s, out["d_s0"],
                        d["cu"], d["cu_host"] if host_cu else None, None, scale, ingate)
    ws = torch.empty(max(rd.bwd_workspace_bytes(prm), 256), dtype=torch.uint8, device="cuda")
    prm.workspace, prm.workspace_bytes = ws.data_ptr(), ws.numel()
    rc = rd.bwd_raw(prm)
    assert rc == rd.OK, rd.status_str(rc)
    assert rd.device_status(ws) == rd.OK
    torch.cuda.synchronize()
    return {n: (None if t is None else host(t)) for n, t in out.items()}


def _check(p, seed, with_state, ingate=rd.INGATE_POW_G, scale=1.0, **kw):
    d_o, d_sT = wl.make_grads(seed, p, with_state)
    got = _run_bwd(p, d_o, d_sT, ingate, scale, **kw)
    ref = orc.ref_bwd(p.q, p.k, p.x, p.y, p.v, d_o, s0=p.s0, dsT=d_sT, cu_seqlens=p.cu_seqlens,
                      scale=scale, ingate=ingate)
    tol = TOL_BF16 if p.dtype == "bf16" else TOL_F32
    errs = {}
    if p.cu_seqlens is None:
        for a, b in PAIRS:
            errs[a] = rel_err(got[a], ref[b])
    else:   # packed: every sequence against its own scale, empty ones have nothing to compare
        cu = p.cu_seqlens
        for a, b in PAIRS:
            errs[a] = max([rel_err(got[a][:, :, cu[n]:cu[n + 1]], ref[b][:, :, cu[n]:cu[n + 1]])
                           for n in range(len(cu) - 1) if cu[n + 1] > cu[n]] or [0.0])
    if got["d_s0"] is not None:
        errs["d_s0"] = rel_err(got["d_s0"], ref["ds0"])
    assert all(e <= tol for e in errs.values()), (p.name, errs)
    return errs


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,H,T,with_state", [
    (1, 1, 1, True),        # a single step
    (2, 2, 16, False),      # exactly one chunk, zero initial state, no state gradient
    (1, 2, 37, True),       # ragged tail
    (2, 3, 150, True),      # several chunks and a ragged tail
])
def test_bwd_matches_oracle(dtype, B, H, T, with_state):
    p = wl.make_prefill(100 + T, B, H, T, 128, 256, dtype, gate_mean=-3.0,
                        s0_std=0.1 if with_state else None, name=f"bwd_{dtype}_{T}")
    _check(p, 200 + T, with_state, scale=0.5)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_bwd_alternate_input_gate_and_strong_decay(dtype):
    # gate pre-activations around +2: decays of e^-1 per step and more, cumulative exponents far
    # below the range of a factored form; every exponential here has a non-positive argument
    p = wl.make_prefill(301, 1, 2, 90, 128, 256, dtype, gate_mean=2.0, s0_std=0.1, name="bwd_strong")
    _check(p, 302, True, ingate=rd.INGATE_POW_SIGMOID)
    _check(p, 303, True, ingate=rd.INGATE_POW_G)
    # pre-activations around +12: a chunk of 16 steps decays by far more than e^-60, which the
    # kernel answers with its pair-by-pair form; milder chunks of the same call take the factored one
    p = wl.make_prefill(304, 1, 2, 70, 128, 256, dtype, gate_mean=12.0, s0_std=0.1, name="bwd_very_strong")
    p.x[:, :, 32:48] = wl.make_prefill(305, 1, 2, 16, 128, 256, dtype, gate_mean=-3.0).x
    _check(p, 306, True, ingate=rd.INGATE_POW_G)
    _check(p, 307, True, ingate=rd.INGATE_POW_SIGMOID)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_bwd_packed_sequences(dtype):
    lens = [40, 0, 1, 16, 77, 3]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    p = wl.make_prefill(401, 1, 2, int(cu[-1]), 128, 256, dtype, s0_std=0.1, cu_seqlens=cu,
                        name="bwd_packed")
    errs = _check(p, 402, True)
    assert "d_s0" in errs
    _check(p, 403, True, host_cu=False, want_d_s0=False)


def test_bwd_bad_cu_seqlens_reported_by_the_device():
    import torch
    cu = np.array([0, 30, 20, 64], dtype=np.int32)          # decreasing
    p = wl.make_prefill(501, 1, 1, 64, 128, 256, "bf16", name="bwd_badcu")
    d = prefill_to_device(p)
    d_o, _ = wl.make_grads(502, p, False)
    outs = [torch.zeros_like(d["q"]) for _ in range(4)] + [torch.zeros_like(d["v"])]
    prm = rd.bwd_params(d["q"], d["k"], d["x"], d["y"], d["v"], dev(d_o, "bf16"), *outs,
                        cu_seqlens=torch.from_numpy(cu).cuda())
    ws = torch.empty(rd.bwd_workspace_bytes(prm), dtype=torch.uint8, device="cuda")
    prm.workspace, prm.workspace_bytes = ws.data_ptr(), ws.numel()
    assert rd.bwd_raw(prm) == rd.OK                          # no host copy: found on the device
    assert rd.device_status(ws) == rd.ERR_SEQLENS
    torch.cuda.synchronize()


def test_bwd_config1_shape_sampled_heads():
    """The layer-prefill shape (B=4, H=16, T=2048) in one call; the oracle checks two heads."""
    import torch
    p = wl.config(1)
    d_o, d_sT = wl.make_grads(601, p, True)
    got = _run_bwd(p, d_o, d_sT, rd.INGATE_POW_G, 1.0)
    for name in got:
        assert np.all(np.isfinite(got[name])), name
    for b, h in ((0, 3), (3, 15)):
        sl = (slice(b, b + 1), slice(h, h + 1))
        ref = orc.ref_bwd(p.q[sl], p.k[sl], p.x[sl], p.y[sl], p.v[sl], d_o[sl], dsT=d_sT[sl])
        for a, r in PAIRS:
            assert rel_err(got[a][sl], ref[r]) <= TOL_BF16, (a, b, h)
        assert rel_err(got["d_s0"][sl], ref["ds0"]) <= TOL_BF16


def test_bwd_long_sequence_and_many_packed_sequences():
    # 1000 steps (63 chunks): the suffix sums run over the whole sequence in 16 time segments
    p = wl.make_prefill(701, 1, 2, 1000, 128, 256, "bf16", s0_std=0.1, name="bwd_long")
    _check(p, 702, True)
    # 40 packed sequences of mixed lengths, several of them shorter than a chunk
    lens = list(np.random.default_rng(703).integers(0, 90, 40))
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    p = wl.make_prefill(704, 1, 2, int(cu[-1]), 128, 256, "bf16", s0_std=0.1, cu_seqlens=cu, name="bwd_many")
    _check(p, 705, True)


def test_bwd_segment_wait_that_runs_out_reports_timeout():
    """A long sweep is cut into time segments that run as thread blocks of their own; each waits,
    with a limit, for the one before it.  With the limit at zero the later segments find their
    predecessors unfinished, give up and return: the call reports TIMEOUT, nothing hangs, and the
    next call is clean."""
    import torch
    p = wl.make_prefill(801, 1, 2, 1000, 128, 256, "bf16", s0_std=0.1, name="bwd_wait")
    d = prefill_to_device(p)
    d_o, d_sT = wl.make_grads(802, p, True)
    outs = [torch.zeros_like(d["q"]) for _ in range(4)] + [torch.zeros_like(d["v"])]
    prm = rd.bwd_params(d["q"], d["k"], d["x"], d["y"], d["v"], dev(d_o, "bf16"), *outs,
                        s0=d["s0"], d_sT=torch.from_numpy(d_sT).cuda())
    ws = torch.empty(rd.bwd_workspace_bytes(prm), dtype=torch.uint8, device="cuda")
    prm.workspace, prm.workspace_bytes = ws.data_ptr(), ws.numel()
    rd.test_set_wait_limit(0)
    try:
        assert rd.bwd_raw(prm) == rd.OK
        assert rd.device_status(ws) == rd.ERR_TIMEOUT
    finally:
        rd.test_set_wait_limit(-1)
    torch.cuda.synchronize()
    _check(p, 802, True)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_bwd_packed_sequences_cut_into_time_segments(dtype):
    # long enough on average for the sweeps to be cut into time segments, with an empty sequence,
    # one of two chunks (one row in the second) and ragged tails among them
    lens = [300, 0, 200, 17, 129]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    p = wl.make_prefill(901, 1, 2, int(cu[-1]), 128, 256, dtype, s0_std=0.1, cu_seqlens=cu,
                        name="bwd_packed_segments")
    _check(p, 902, True)
    _check(p, 903, False, host_cu=False, want_d_s0=False)


@pytest.mark.parametrize("T", [2, 63, 64, 65, 129, 520])
@pytest.mark.parametrize("strong", [False, True])
def test_bwd_bf16_tile_edges_and_cut_tiles(T, strong):
    """Edges of the 64-row tiles, time segments (520 rows), and tiles that strong decays cut into
    several chunks: single steps of e^-60 and more among mild ones, in some channels only.  Bar of
    this file for bf16.

    A strong step's dx is w tau sigmoid(x)/g - dla tau sigmoid(x) where dla, nearly zero, is a
    difference of sums as large as w; the states are read as tf32 (2^-11), so dx carries an error of up
    to 2^-11 g of the size of its first term: 4e-2 at g = 80, beyond the bar where such steps are all
    there is.  Two rows therefore take g = 20 (1e-2); longer sequences have mild rows, whose dx is
    larger and sets the scale."""
    p = wl.make_prefill(1000 + T, 1, 2, T, 128, 256, "bf16", s0_std=0.1, name=f"bwd_tile_{T}")
    if strong:
        p.x[:, :, T // 3:T // 3 + 7, ::5] = 80.0 if T > 2 else 20.0     # softplus(80) sigmoid(4) = 78.6 per step
        p.y[:, :, T // 3:T // 3 + 7, ::5] = 4.0
    _check(p, 1100 + T, True, scale=0.5)


@pytest.mark.parametrize("n_seq,shortest,longest", [(30, 62, 148), (7, 50, 600)])
def test_bwd_packed_pieces_that_follow_one_another_on_a_block(n_seq, shortest, longest):
    """More sweeps than thread blocks, of one to a few tiles and of every kind in turn: what a block's
    roles hand over from the end of one sweep to the beginning of the next.  Nothing depends on which
    block runs which sweep, so repeated calls agree bit for bit; the first against the oracle."""
    lens = np.random.default_rng(n_seq).integers(shortest, longest + 1, n_seq)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    p = wl.make_prefill(1200 + n_seq, 1, 16, int(cu[-1]), 128, 256, "bf16", cu_seqlens=cu, s0_std=0.1, name=f"bwd_pieces_{n_seq}")
    _check(p, 1201, True)
    d_o, d_sT = wl.make_grads(1201, p, True)
    first = _run_bwd(p, d_o, d_sT, rd.INGATE_POW_G, 1.0)
    for _ in range(12):
        again = _run_bwd(p, d_o, d_sT, rd.INGATE_POW_G, 1.0)
        assert all(np.array_equal(first[n], again[n]) for n in first)


def test_bwd_bad_cu_seqlens_with_overlapping_ranges_stays_in_the_workspace():
    """Ranges that overlap have more tiles than the workspace has places for.  At this length the list of
    tiles ends the workspace (its few words per tile outgrow the room for states), so that entries beyond
    the list would land in the guard behind it."""
    import torch
    T, N, guard = 160000, 3, 1 << 20
    q, k, x, y = (torch.zeros((1, 1, T, 128), dtype=torch.bfloat16, device="cuda") for _ in range(4))
    v, d_o = (torch.zeros((1, 1, T, 256), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    out = [torch.empty_like(t) for t in (q, k, x, y, v)]
    cu = torch.tensor([0, T, 0, T], dtype=torch.int32, device="cuda")
    prm = rd.bwd_params(q, k, x, y, v, d_o, *out, cu_seqlens=cu)
    need = rd.bwd_workspace_bytes(prm)
    ws = torch.full((need + guard,), 0xA5, dtype=torch.uint8, device="cuda")
    prm.workspace, prm.workspace_bytes = ws.data_ptr(), need
    assert rd.bwd_raw(prm) == rd.OK and rd.device_status(ws) == rd.ERR_SEQLENS
    assert bool((ws[need:] == 0xA5).all())


@pytest.mark.parametrize("N", [513, 4200])                    # sorted by length; too many to sort
def test_bwd_bf16_more_packed_sequences_than_a_block_has_threads(N):
    lens = np.random.default_rng(N).integers(0, 3, N)
    lens[N // 2:N // 2 + 40] = 0
    lens[[N // 3, N // 5]] = 200, 70
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    _check(wl.make_prefill(1300 + N, 1, 1, int(cu[-1]), 128, 256, "bf16", s0_std=0.1, cu_seqlens=cu, name=f"bwd_many_{N}"),
           1301, True)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("bad", [("v",), ("d_o",), ("q", "k", "x", "y")])
@pytest.mark.parametrize("B,H,T,packed,gate_mean", [(2, 2, 200, None, -3.0), (1, 3, 63, None, -3.0), (1, 2, 200, None, 1.5),
                                                    (1, 40, 130, None, -3.0), (1, 3, 0, (100, 40, 60), -3.0),
                                                    (1, 2, 0, (65, 1, 64), 1.5)])
def test_bwd_neighbours_nan_stays_out(value, bad, B, H, T, packed, gate_mean):
    """The first rows of every head but the first (packed: of every sequence but the first) get NaN or infinities;
    gradients of what lies before them stay bit for bit what they were.  Tiles whole and cut into chunks, sweeps
    whole and cut in two."""
    import torch
    cu = None if packed is None else np.concatenate([[0], np.cumsum(packed)]).astype(np.int32)
    p = wl.make_prefill(1400, B, H, T if cu is None else int(cu[-1]), 128, 256, "bf16", gate_mean=gate_mean, s0_std=0.2, cu_seqlens=cu)
    g_o, g_s = wl.make_grads(1401, p, True)
    d = prefill_to_device(p)
    d["d_o"] = dev(g_o, p.dtype)
    got = []
    for spoilt in (False, True):
        for name in bad if spoilt else ():
            if cu is None: d[name][:, 1:, :3] = value
            else: d[name][:, :, int(cu[1]):int(cu[1]) + 3] = value
        g = rd.ddts_bwd(*(d[n] for n in ("q", "k", "x", "y", "v", "d_o")), d["s0"], torch.from_numpy(g_s).cuda(), cu_seqlens=d["cu"],
                        want_d_s0=True)
        if cu is None: got.append([t[:, 0] for t in g.values()])
        else: got.append([g["d_s0"][0]] + [t[:, :, :int(cu[1])] for n, t in g.items() if n != "d_s0"])
    for clean, spoilt in zip(*got):
        assert torch.isfinite(clean).all() and torch.equal(clean, spoilt)
