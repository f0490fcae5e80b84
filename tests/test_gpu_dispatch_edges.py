"""Parity at the sizes where a dispatch rule changes its mind or a tile is ragged: one row past a tile, the last size of a
split, head counts that are not powers of two.  Tolerances are those of the files that cover the same entry points."""
import numpy as np
import pytest
import torch

from oracle import dsla_oracle as orc

pytestmark = pytest.mark.gpu
BF = torch.bfloat16


# split 8 (few tiles), 4 (19..37 tiles), 2 (38..74), none; H = 40: twenty 16-byte pieces per row; H = 8: four
@pytest.mark.parametrize("T,H,D_model", [(127, 40, 2048), (18 * 128 + 1, 8, 2048), (37 * 128, 16, 1024), (38 * 128 - 1, 24, 512),
                                         (75 * 128 - 5, 8, 512), (200, 96, 1024)])
def test_gate_project_cluster_splits(T, H, D_model):
    import paper_2506_09316_b200 as dsla
    rng = np.random.default_rng(5100 + T)
    x = torch.from_numpy(rng.normal(size=(T, D_model)).astype(np.float32)).to(BF)
    w = torch.from_numpy((rng.normal(size=(2 * H, D_model)) * (2.0 / np.sqrt(D_model))).astype(np.float32)).to(BF)
    b = torch.from_numpy(rng.normal(size=2 * H).astype(np.float32) * 2.0)
    band = 64
    gh, gr = (torch.full((T + band, H), 7.0, device="cuda") for _ in range(2))
    for _ in range(2):          # back to back: the second launch overlaps the first one's tail
        dsla.dsla_gate_project(x.cuda(), w.cuda(), b.cuda(), g_hist=gh[:T], g_rec=gr[:T])
    torch.cuda.synchronize()
    assert dsla.dsla_gate_project_last_error() == dsla.DSLA_OK
    rows = np.unique(np.concatenate([np.arange(min(T, 160)), np.arange(max(0, T - 160), T)]))
    ref = orc.gate_project(x[rows].double().numpy(), w.double().numpy().T, b.double().numpy())
    got = np.concatenate([gh[:T].double().cpu().numpy()[rows], gr[:T].double().cpu().numpy()[rows]], axis=1)
    assert np.max(np.abs(got - ref)) <= 2e-5
    assert bool((gh[:T] <= 1.0).all()) and bool((gr[:T] <= 1.0).all())      # every row written
    assert bool((gh[T:] == 7.0).all()) and bool((gr[T:] == 7.0).all())      # and none past the end


# CUDA-core chunkwise prefill: 8, 4, 2 and 1 segments per sequence (one cluster each), segments of one chunk and of several, a last
# segment of one token, segments without a chunk (a packed batch's short sequences), and an empty sequence in a cluster
@pytest.mark.parametrize("lens,H,d,dtype,chunk", [
    ((512,), 4, 64, torch.float32, 64), ((513,), 2, 128, torch.float32, 64), ((1100,), 9, 64, torch.float32, 64),
    ((1025,), 18, 64, BF, 32), ((260,), 80, 64, torch.float32, 64), ((700, 0, 65, 1), 2, 64, torch.float32, 64),
    ((129, 64, 300), 1, 128, BF, 16)])
@pytest.mark.parametrize("resume", [False, True])
def test_simt_prefill_segments(lens, H, d, dtype, chunk, resume):
    from paper_2506_09316_b200 import inputs as gen
    from util import TOL, gpu_prefill, oracle_prefill, rel_err
    inp = gen.make_packed(5200 + sum(lens) + H, lens, H, d, dtype)
    inp.g_rec[::37] = 0.0                   # exact zeros inside and at the edges of segments
    inp.g_hist[100::211] = 0.0
    slots = np.random.default_rng(1).permutation(len(lens) + 1)[:len(lens)].astype(np.int32)
    state0 = gen.make_states(5201, len(lens) + 1, H, d, d, std=0.5).numpy() if resume else None
    o, S = gpu_prefill(inp, num_slots=len(lens) + 1, state0=state0, slots=slots, chunk=chunk, impl="simt", scale=0.8)
    start = np.zeros(S.shape) if state0 is None else state0.astype(np.float64)
    o_ref, S_ref = oracle_prefill(inp, state0=start, slots=slots, scale=0.8)
    assert rel_err(o, o_ref) <= TOL[dtype] and rel_err(S[slots], S_ref[slots]) <= TOL[torch.float32]


# Short sequences take chunks of 16 and 32 tokens: both sides of each line, a packed batch whose longest sequence decides
@pytest.mark.parametrize("lens,H,d", [((1,), 2, 64), ((16,), 3, 64), ((17,), 2, 128), ((32,), 4, 128), ((33,), 2, 64), ((9, 0, 31), 2, 64)])
def test_simt_prefill_short(lens, H, d):
    from paper_2506_09316_b200 import inputs as gen
    from util import TOL, gpu_prefill, oracle_prefill, rel_err
    inp = gen.make_packed(5600 + sum(lens) + d, lens, H, d, torch.float32)
    inp.g_rec[5::7] = 0.0
    slots = np.arange(len(lens), dtype=np.int32)
    state0 = gen.make_states(5601, len(lens), H, d, d, std=0.5).numpy()
    o, S = gpu_prefill(inp, num_slots=len(lens), state0=state0, slots=slots, scale=0.8)
    o_ref, S_ref = oracle_prefill(inp, state0=state0.astype(np.float64), slots=slots, scale=0.8)
    assert rel_err(o, o_ref) <= TOL[torch.float32] and rel_err(S, S_ref) <= TOL[torch.float32]


# Gates per key channel on the tensor cores: whole and ragged chunks of 32 tokens, one token past a block, several segments and one (too few
# chunks or too many heads), exact zeros and ones, sequences shorter than a segment
@pytest.mark.parametrize("lens,H,resume", [((1,), 2, False), ((16,), 1, True), ((17,), 3, False), ((32,), 2, True), ((33, 31, 0, 64), 2, True),
                                           ((257,), 2, False), ((515, 40, 260), 1, True), ((1030,), 37, False), ((300,), 80, True)])
@pytest.mark.parametrize("pattern", ["mix", "zeros", "ones"])
def test_channel_prefill_tensor(lens, H, resume, pattern):
    from paper_2506_09316_b200 import inputs as gen
    from util import TOL, gpu_prefill, oracle_prefill, rel_err
    if pattern != "mix" and sum(lens) > 300:
        pytest.skip("the long cases run with mixed gates")
    inp = gen.make_packed(5300 + sum(lens) + H, lens, H, 128, BF)
    rng = np.random.default_rng(5301)
    shape = (inp.T_total, H, 128)
    for name, mu in (("g_hist", 5.0), ("g_rec", 1.0)):
        g = 1.0 / (1.0 + np.exp(-rng.normal(mu, 2.0, size=shape)))
        u = rng.uniform(size=shape)
        g = np.where(u < 0.02, 0.0, np.where(u > 0.98, 1.0, g)) if pattern == "mix" else np.full(shape, 0.0 if pattern == "zeros" else 1.0)
        setattr(inp, name, torch.from_numpy(g.astype(np.float32)))
    slots = rng.permutation(len(lens) + 1)[:len(lens)].astype(np.int32)
    state0 = gen.make_states(5302, len(lens) + 1, H, 128, 128, std=0.5).numpy() if resume else None
    start = np.zeros((len(lens) + 1, 2, H, 128, 128)) if state0 is None else state0.astype(np.float64)
    o_ref, S_ref = oracle_prefill(inp, state0=start, slots=slots, scale=0.7)
    o, S = gpu_prefill(inp, num_slots=len(lens) + 1, state0=state0, slots=slots, scale=0.7)
    # states: fp32 sums of exact products (three bf16 terms of an fp32 factor); outputs: one bf16 rounding (2^-9 of the value)
    assert rel_err(S[slots], S_ref[slots]) <= 1e-5
    assert rel_err(o, o_ref) <= 4e-3


# Vector gates cut a sequence into as many segments as the workspace has room for: none, a misaligned one, room for two, for all that
# dsla_prefill_workspace_bytes gives (four here), and the array inside the library; fresh and continued (the slot pushed through the first summary).
@pytest.mark.parametrize("resume", [False, True])
def test_channel_prefill_workspaces(resume):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    from util import oracle_prefill, rel_err
    T, H, stride = 1100, 2, (2 * 128 * 128 + 2 * 128) * 4
    inp = gen.make_packed(5390, [T], H, 128, BF)
    rng = np.random.default_rng(5391)
    for name, mu in (("g_hist", 6.0), ("g_rec", 1.0)):
        setattr(inp, name, torch.from_numpy((1.0 / (1.0 + np.exp(-rng.normal(mu, 0.5, size=(T, H, 128))))).astype(np.float32)))
    state0 = gen.make_states(5392, 1, H, 128, 128, std=0.5)
    o_ref, S_ref = oracle_prefill(inp, state0=state0.double().numpy() if resume else np.zeros(tuple(state0.shape)))
    dv, st = inp.to("cuda"), dsla.dsla_state_alloc(1, H, 128, 128)
    full = dsla.dsla_prefill_workspace_bytes(T, 1, T, H, 128, dense_T=T, gate_layout=dsla.DSLA_GATE_PER_KEY_CHANNEL)
    assert full == 4 * H * stride
    room = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    forms = [("none", room[:0], 1), ("too small", room[:2 * H * stride - 1], 1), ("misaligned", room[8:], 1), ("two", room[:2 * H * stride], 2),
             ("full", room[:full], 2), ("the binding's", None, 2), ("static", None, 2)]
    results = {}
    for name, ws, launches in forms:
        st.tensor.copy_(state0)
        before = dsla.dsla_launch_count()
        if name == "static":
            o = dsla.dsla_prefill_static_ws(dv.q, dv.k, dv.v, dv.g_hist, dv.g_rec, dv.gamma, st, use_initial_state=resume)
        else:
            o = dsla.dsla_prefill(dv.q, dv.k, dv.v, dv.g_hist, dv.g_rec, dv.gamma, st, use_initial_state=resume, workspace=ws)
        assert dsla.dsla_launch_count() - before == launches, name
        assert dsla.dsla_state_last_error(st) == dsla.DSLA_OK
        assert rel_err(o.double().cpu().numpy(), o_ref) <= 4e-3 and rel_err(st.tensor.double().cpu().numpy(), S_ref) <= 1e-5, name
        results[name] = (o, st.tensor.clone())
    for name in ("the binding's", "static"):
        assert all(torch.equal(x, y) for x, y in zip(results[name], results["full"])), name


# The states of the tensor-core kernel for vector gates are fp32 sums like those of the token-by-token kernel, and no further from the
# exact ones: 260 tokens in one segment, 2000 in several.
@pytest.mark.parametrize("T,H", [(260, 4), (1100, 40), (2000, 4)])
def test_channel_prefill_state_precision(T, H):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    from util import oracle_prefill
    inp = gen.make_packed(5350 + T, [T], H, 128, BF)
    rng = np.random.default_rng(5351)
    for name, mu in (("g_hist", 6.0), ("g_rec", 1.0)):
        g = 1.0 / (1.0 + np.exp(-rng.normal(mu, 0.5, size=(T, H, 128))))
        setattr(inp, name, torch.from_numpy(g.astype(np.float32)))
    dv, st = inp.to("cuda"), dsla.dsla_state_alloc(1, H, 128, 128)
    _, S_ref = oracle_prefill(inp, state0=np.zeros((1, 2, H, 128, 128)))
    off = {}
    for impl in ("auto", "simt"):
        dsla.dsla_prefill(dv.q, dv.k, dv.v, dv.g_hist, dv.g_rec, dv.gamma, st, impl=impl)
        off[impl] = np.linalg.norm(st.tensor.double().cpu().numpy() - S_ref) / np.linalg.norm(S_ref)
    assert off["auto"] <= off["simt"], off


# What a token adds to a state, w k^T v, is rounded to bf16 once (w v; the weight itself has 16 bits): at most 2^-9 of it, whether the
# sequence is one chunk, one segment or several.
@pytest.mark.parametrize("T,H", [(64, 8), (128, 8), (777, 4), (1500, 150)])
def test_tensor_prefill_state_precision(T, H):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    from util import oracle_prefill
    inp = gen.make_packed(5360 + T, [T], H, 128, BF)
    dv, st = inp.to("cuda"), dsla.dsla_state_alloc(1, H, 128, 128)
    dsla.dsla_prefill(dv.q, dv.k, dv.v, dv.g_hist, dv.g_rec, dv.gamma, st, impl="tensor")
    _, S_ref = oracle_prefill(inp, state0=np.zeros((1, 2, H, 128, 128)))
    for i in range(2):
        S, ref = st.tensor[:, i].double().cpu().numpy(), S_ref[:, i]
        assert np.linalg.norm(S - ref) <= 2.0 ** -9 * np.linalg.norm(ref)


# The order in which a packed batch is visited: found inside the kernel (up to 64 sequences, one and two per lane) and by a kernel of its
# own (more); ties and empty sequences, whole sequences and split ones
@pytest.mark.parametrize("N,H,top", [(2, 3, 500), (31, 5, 90), (33, 4, 200), (64, 3, 70), (65, 3, 70)])
def test_packed_order(N, H, top):
    from paper_2506_09316_b200 import inputs as gen
    from util import TOL, gpu_prefill, oracle_prefill, rel_err
    rng = np.random.default_rng(5400 + N)
    lens = [int(x) for x in rng.integers(0, top, N)]
    lens[N // 2] = lens[0]
    inp = gen.make_packed(5401 + N, lens, H, 128, BF)
    slots = rng.permutation(N + 1)[:N].astype(np.int32)
    state0 = gen.make_states(5402, N + 1, H, 128, 128, std=0.5).numpy()
    o, S = gpu_prefill(inp, num_slots=N + 1, state0=state0, slots=slots, impl="tensor")
    o_ref, S_ref = oracle_prefill(inp, state0=state0.astype(np.float64), slots=slots)
    assert rel_err(o, o_ref) <= TOL[BF] and rel_err(S[slots], S_ref[slots]) <= TOL[BF]


# Segments on the CTAs of a cluster, all of which leave together: batches in which segments have no chunk, one chunk or several, and a
# sequence none at all, one launch behind the other; every run gives the same bits.
@pytest.mark.parametrize("lens,H", [((1500, 0, 64, 777, 130), 2), ((257,), 1), ((4096, 1), 3), ((385, 2000), 17)])
@pytest.mark.parametrize("resume", [False, True])
def test_split_clusters_leave_together(lens, H, resume):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    from util import TOL, oracle_prefill, rel_err
    inp = gen.make_packed(5450 + sum(lens), lens, H, 128, BF)
    state0 = gen.make_states(5451, len(lens), H, 128, 128, std=0.5)
    dv, st, runs = inp.to("cuda"), dsla.dsla_state_alloc(len(lens), H, 128, 128), []
    for _ in range(20):
        st.tensor.copy_(state0)
        o = dsla.dsla_prefill(dv.q, dv.k, dv.v, dv.g_hist, dv.g_rec, dv.gamma, st, cu_seqlens=dv.cu_seqlens, max_seqlen=max(lens),
                              use_initial_state=resume, impl="tensor")
        runs.append((o, st.tensor.clone()))
    assert dsla.dsla_state_last_error(st) == dsla.DSLA_OK
    assert all(torch.equal(o, runs[0][0]) and torch.equal(S, runs[0][1]) for o, S in runs[1:])
    o_ref, S_ref = oracle_prefill(inp, state0=state0.double().numpy() if resume else np.zeros(tuple(state0.shape)))
    assert rel_err(runs[0][0].double().cpu().numpy(), o_ref) <= TOL[BF]
    assert rel_err(runs[0][1].double().cpu().numpy(), S_ref) <= TOL[BF]


# The tiles of a sequence's last chunk also hold the first tokens of the next sequence, which may be anything: with infinities and NaN in q, k
# and v of every other sequence, a sequence comes out as it does alone.
@pytest.mark.parametrize("lens,H", [((64, 90), 2), ((100, 1), 3), ((5, 700, 129), 2), ((300, 40), 150), ((1, 200), 1)])
@pytest.mark.parametrize("form", ["dual", "four", "channel", "f32"])
def test_neighbour_sequences_do_not_leak(lens, H, form):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    inp = gen.make_packed(5470 + sum(lens), lens, H, 128, torch.float32 if form == "f32" else BF)
    if form == "channel":
        rng = np.random.default_rng(5471)
        for name in ("g_hist", "g_rec"):
            setattr(inp, name, torch.from_numpy(rng.uniform(0.3, 1.0, size=(inp.T_total, H, 128)).astype(np.float32)))
    d = inp.to("cuda")
    gates, w = torch.stack([d.g_hist, d.g_rec, d.g_hist, d.g_rec]), torch.full((H, 4), 0.25, device="cuda")
    cu = [0] + list(np.cumsum(lens))

    def run(q, k, v):
        st = dsla.dsla_state_alloc_n(len(lens), 4, H, 128, 128) if form == "four" else dsla.dsla_state_alloc(len(lens), H, 128, 128)
        kw = dict(cu_seqlens=d.cu_seqlens, max_seqlen=max(lens))
        if form == "four":
            o = dsla.dsla_nstate_prefill(q, k, v, gates, w, st, **kw)
        else:
            o = dsla.dsla_prefill(q, k, v, d.g_hist, d.g_rec, d.gamma, st, **kw)
        assert dsla.dsla_state_last_error(st) == dsla.DSLA_OK
        return o, st.tensor

    o0, S0 = run(d.q, d.k, d.v)
    assert bool(torch.isfinite(o0).all()) and bool(torch.isfinite(S0).all())
    for keep in range(len(lens)):
        dirty = [x.clone() for x in (d.q, d.k, d.v)]
        for x, bad in zip(dirty, (float("nan"), float("inf"), float("nan"))):
            x[:cu[keep]] = bad
            x[cu[keep + 1]:] = bad
        o, S = run(*dirty)
        assert torch.equal(o[cu[keep]:cu[keep + 1]], o0[cu[keep]:cu[keep + 1]]) and torch.equal(S[keep], S0[keep])


# Token by token, an infinity or NaN in v reaches no output before it.  Its chunk's products are matrix products with zeros for the tokens
# before it, and 0 * inf is not 0: at the first and last rows of a chunk of 32 and of its blocks of 16, in the ragged last chunk, in the
# last one but one, in a later segment; o before it and every other column as without it, the states non-finite in that column alone.
@pytest.mark.parametrize("T,H,at", [(40, 2, (0,)), (64, 3, (31, 40)), (97, 1, (16, 47, 96)), (700, 2, (350, 699)), (333, 160, (200,))])
@pytest.mark.parametrize("bad", [float("nan"), float("-inf")])
def test_channel_prefill_is_causal_in_v(T, H, at, bad):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    inp = gen.make_packed(5480 + T, [T], H, 128, BF)
    rng = np.random.default_rng(5481)
    for name in ("g_hist", "g_rec"):
        setattr(inp, name, torch.from_numpy(rng.uniform(0.3, 1.0, size=(T, H, 128)).astype(np.float32)))
    d = inp.to("cuda")

    def run(v):
        st = dsla.dsla_state_alloc(1, H, 128, 128)
        o = dsla.dsla_prefill(d.q, d.k, v, d.g_hist, d.g_rec, d.gamma, st)
        assert dsla.dsla_state_last_error(st) == dsla.DSLA_OK
        return o, st.tensor

    o0, S0 = run(d.v)
    for t in at:
        v, col = d.v.clone(), (37 * t) % 128
        v[t, H - 1, col] = bad
        o, S = run(v)
        hit = torch.zeros_like(o, dtype=torch.bool)
        hit[t:, H - 1, col] = True
        assert not bool(torch.isfinite(o[hit]).any())
        # the chunk's other outputs add fp32 scores instead of two bf16 terms of them: one rounding of the output apart
        assert bool(torch.isfinite(o[~hit]).all())
        assert float((o.float() - o0.float())[~hit].abs().max()) <= 2.0 ** -8 * float(o0.float().abs().max())
        rest = [c for c in range(128) if c != col]
        assert torch.equal(S[:, :, :, :, rest], S0[:, :, :, :, rest]) and not bool(torch.isfinite(S[0, :, H - 1, :, col]).any())


# Pairs of states side by side in a cluster: two and four pairs, with one segment per sequence and with several (clusters of up to 16),
# whole chunks and ragged ones, a batch of which one sequence is empty and one shorter than a segment; 75 heads: one pair at a time
@pytest.mark.parametrize("n,lens,H,resume", [(4, (100,), 3, False), (8, (128,), 2, True), (4, (129,), 74, True), (4, (1500, 0, 64, 777), 2, True),
                                             (8, (1153,), 3, False), (8, (640, 300), 5, True), (4, (1024,), 32, False), (4, (257,), 75, False)])
def test_nstate_pairs_in_one_cluster(n, lens, H, resume):
    import paper_2506_09316_b200 as dsla
    from paper_2506_09316_b200 import inputs as gen
    from util import TOL, rel_err
    rng = np.random.default_rng(5500 + n + sum(lens))
    inp = gen.make_packed(5501 + H, lens, H, 128, BF)
    gates = (1.0 / (1.0 + np.exp(-rng.normal(3.0, 1.5, size=(n, inp.T_total, H))))).astype(np.float32)
    gates[:, 60, :] = 0.0
    w = rng.normal(size=(H, n)).astype(np.float32)
    st0 = (rng.normal(size=(len(lens), n, H, 128, 128)) * 0.3).astype(np.float32)
    dv, g, wd = inp.to("cuda"), torch.from_numpy(gates).cuda(), torch.from_numpy(w).cuda()
    st, outs = dsla.dsla_state_alloc_n(len(lens), n, H, 128, 128), []
    for _ in range(2):          # back to back; the order in which the pairs add to o is fixed, so the second run gives the same bits
        st.tensor.copy_(torch.from_numpy(st0))
        outs.append(dsla.dsla_nstate_prefill(dv.q, dv.k, dv.v, g, wd, st, cu_seqlens=dv.cu_seqlens, max_seqlen=max(lens),
                                             use_initial_state=resume, scale=0.8))
    torch.cuda.synchronize()
    assert dsla.dsla_state_last_error(st) == dsla.DSLA_OK
    assert torch.equal(outs[0], outs[1])
    f = inp.as_f64()
    start = st0.astype(np.float64) if resume else np.zeros(st0.shape)
    o_ref, S_ref = orc.prefill_n(f["q"], f["k"], f["v"], gates, w, f["cu_seqlens"], scale=0.8, state=start)
    assert rel_err(outs[0].double().cpu().numpy(), o_ref) <= TOL[BF] * (1.5 if n == 8 else 1.0)
    assert rel_err(st.tensor.double().cpu().numpy(), S_ref) <= TOL[BF]
