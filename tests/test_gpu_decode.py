"""GPU parity: qjoint_logprobs, the prediction/joint path of config 2 and the fused beam
search (dr_fusion_beam_step) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2206_07882_b200 import synth
from _parity import gpu_codes, pack_codes, to_act, written_late

pytestmark = pytest.mark.gpu

LP_ATOL = 1e-5     # log-softmax: fp32 reduction on the GPU vs double in the oracle, |lp| <= ~20


@pytest.fixture(scope="module")
def Bd():
    from paper_2206_07882_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("N,V,D,Hp,zb,prep", [(5, 64, 32, 64, 4, False), (70, 1024, 256, 1024, 4, False),
                                                  (33, 200, 64, 96, 8, False),
                                                  # tensor-core path: fused head (D = 256), ragged last row tile;
                                                  # GEMM + row log-softmax (D = 64); 8-bit output layer
                                                  (200, 1024, 256, 1024, 4, True), (130, 96, 64, 128, 4, True),
                                                  (257, 992, 256, 256, 8, True),
                                                  # one row tile, mostly empty
                                                  (1, 1024, 256, 256, 4, True), (70, 96, 64, 128, 8, True)])
def test_joint_logprobs(Bd, N, V, D, Hp, zb, prep):
    dw = synth.decoder(seed=5, V=V, E=32, Hp=Hp, D=D, Hs=32, Ht=32, out_bits=zb)
    dec = O.Decoder(dw)
    st = synth.Stream(9)
    R = 40
    e = st.normal("e", (R, D)).astype(np.float32)
    fi = st.integers("fi", (N,), 0, R - 1).astype(np.int32)
    hid = O.act_symmetric(1.0, 4)
    pq = st.integers("pq", (N, Hp), -7, 7).astype(np.int16)
    p = O.linear(O.Linear(dw.pred.proj), pq, hid)
    want = O.joint(dec, e[fi], p)
    dd = Bd.Decoder(dw)
    if prep:
        dd.pred_proj.prepare()
        dd.joint_out.prepare()
    n0 = Bd.launch_count()
    got = Bd.qjoint_logprobs(torch.from_numpy(e).cuda(), torch.from_numpy(fi).cuda(), pack_codes(pq, hid),
                             to_act(hid), dd.pred_proj, dd.z_act, dd.joint_out).cpu().numpy()
    assert Bd.launch_count() - n0 == ((3 if D == 256 else 4) if prep else 4)
    assert np.abs(got - want).max() <= LP_ATOL
    np.testing.assert_allclose(np.exp(got.astype(np.float64)).sum(1), 1.0, atol=1e-5)


@pytest.mark.parametrize("N,D", [(3, 256), (40, 64), (130, 256)])
def test_joint_rows_without_a_frame(Bd, N, D):
    # a negative frame index stands for a frame of zeros, with prepared weights as without
    dw = synth.decoder(seed=7, V=64, E=32, Hp=128, D=D, Hs=32, Ht=32)
    st = synth.Stream(11)
    e = st.normal("e", (9, D)).astype(np.float32)
    fi = st.integers("fi", (N,), 0, 8).astype(np.int32)
    fi[[0, N // 2, N - 1]] = -1
    hid = O.act_symmetric(1.0, 4)
    pq = st.integers("pq", (N, 128), -7, 7).astype(np.int16)
    frames = np.where(fi[:, None] >= 0, e[fi], np.float32(0))
    want = O.joint(O.Decoder(dw), frames, O.linear(O.Linear(dw.pred.proj), pq, hid))
    dd = Bd.Decoder(dw)
    for prepare in (False, True):
        if prepare:
            dd.pred_proj.prepare()
            dd.joint_out.prepare()
        got = Bd.qjoint_logprobs(torch.from_numpy(e).cuda(), torch.from_numpy(fi).cuda(), pack_codes(pq, hid), to_act(hid),
                                 dd.pred_proj, dd.z_act, dd.joint_out).cpu().numpy()
        assert np.abs(got - want).max() <= LP_ATOL


def pred_joint_gpu(Bd, dd, e_dev, frame_idx, tokens):
    """Teacher-forced prediction network + joint on the GPU: logp [N,S,V], hq codes [N,S,Hp]."""
    N, S = tokens.shape
    Hp, V = dd.pred_lstm.H, dd.V
    # one-time int8 operands: these calls run on the tensor-core kernels (steps of up to 32 rows on the weight-streaming one)
    dd.pred_lstm.prepare()
    dd.pred_proj.prepare()
    dd.joint_out.prepare()
    hq = torch.zeros((N, Hp // 2), dtype=torch.uint8, device="cuda")
    c = torch.zeros((N, Hp), dtype=torch.float32, device="cuda")
    tok = torch.from_numpy(tokens).cuda()
    fi = torch.from_numpy(frame_idx).cuda()
    out = torch.empty((N, S, V), dtype=torch.float32, device="cuda")
    hqs = []
    for s in range(S):
        r = Bd.qlstm_step(dd.pred_emb_q, dd.pred_emb_act, hq, c, dd.pred_lstm,
                          x_row_idx=tok[:, s].contiguous())
        hq, c = r["hq"], r["c"]
        out[:, s] = Bd.qjoint_logprobs(e_dev, fi[:, s].contiguous(), hq, dd.pred_lstm.hid_act,
                                       dd.pred_proj, dd.z_act, dd.joint_out)
        hqs.append(hq)
    return out, torch.stack(hqs, dim=1)


def test_config2_reduced_all_rows(Bd):
    dw = synth.decoder(seed=2, V=64, E=32, Hp=64, D=32, Hs=32, Ht=32)
    N, S, T, B = 48, 20, 20, 3
    encq_act = O.act_symmetric(1.0, 4)
    frames = synth.enc_frames(2, T, B, 64)
    proj = synth._linear(synth.Stream(2), "enc.proj", 32, 64)
    e = O.linear(O.Linear(proj), O.quantize(frames.astype(np.float32).reshape(T * B, 64), encq_act), encq_act)
    toks = np.concatenate([np.zeros((N, 1), np.int32), synth.labels(2, N, S - 1, 64)], axis=1)
    fi = (np.arange(S, dtype=np.int32)[None, :] * B + (np.arange(N, dtype=np.int32)[:, None] % B)).astype(np.int32)
    want, hq_w, c_w, p_w = O.pred_joint_forced(O.Decoder(dw), e, fi, toks, want_state=True)
    dd = Bd.Decoder(dw)
    got, hq_g = pred_joint_gpu(Bd, dd, torch.from_numpy(e).cuda(), fi, toks)
    np.testing.assert_array_equal(gpu_codes(hq_g.reshape(N * S, -1), 64, encq_act).reshape(N, S, 64), hq_w)
    assert np.abs(got.cpu().numpy() - want).max() <= LP_ATOL


def test_config2_full_size_sampled_rows(Bd):
    # 256 hypothesis rows x 300 steps; vocabulary 1024, embedding 256, prediction LSTM 1024,
    # joint 1280 -> 256 -> 1024.  The oracle recomputes 3 of the 256 rows (rows are independent).
    dw = synth.decoder(seed=2)
    B, W, T, S = 16, 16, 300, 300
    N = B * W
    act = O.act_symmetric(1.0, 4)
    frames = synth.enc_frames(2, T, B, 1280)
    proj = synth._linear(synth.Stream(2), "enc.proj", 256, 1280)
    dproj = Bd.DeviceLinear(proj)
    fq = Bd.quantize_pack_int4(torch.from_numpy(frames).cuda().reshape(T * B, 1280), to_act(act))
    e_dev = Bd.q4_linear_forward(fq, to_act(act), dproj)
    toks = np.concatenate([np.zeros((N, 1), np.int32), synth.labels(2, N, S - 1, 1024)], axis=1)
    fi = (np.arange(S, dtype=np.int32)[None, :] * B + (np.arange(N, dtype=np.int32)[:, None] // W)).astype(np.int32)
    dd = Bd.Decoder(dw)
    got, hq_g = pred_joint_gpu(Bd, dd, e_dev, fi, toks)
    rows = [0, 117, 255]
    e = e_dev.cpu().numpy()
    # the projected frames themselves: bit-exact against the oracle on the frames those rows use
    used = np.unique(fi[rows])
    e_ref = O.linear(O.Linear(proj), O.quantize(frames.astype(np.float32).reshape(T * B, 1280)[used], act), act)
    np.testing.assert_array_equal(e[used], e_ref)
    want, hq_w, _, _ = O.pred_joint_forced(O.Decoder(dw), e, fi[rows], toks[rows], want_state=True)
    np.testing.assert_array_equal(gpu_codes(hq_g[rows].reshape(len(rows) * S, -1), 1024, act).reshape(len(rows), S, 1024), hq_w)
    assert np.abs(got[rows].cpu().numpy() - want).max() <= LP_ATOL


def run_search(Bd, dw, e, utts=None, tensor_cores=True):
    dd = Bd.Decoder(dw, tensor_cores=tensor_cores)
    T, B, D = e.shape
    tokens, lens, scores = dd.decode(torch.from_numpy(e).cuda())
    torch.cuda.synchronize()
    assert dd.tensors["status"].item() == 0
    ref = O.alsd(O.Decoder(dw), e, utts=utts)
    return dd, tokens.cpu().numpy(), lens.cpu().numpy(), scores.cpu().numpy(), ref


def compare_search(dd, tokens, lens, scores, ref, utts, T, U, W, min_same=0.99):
    IT = T + U
    bp_parent = dd.tensors["bp_parent"].cpu().numpy()[:IT]
    bp_token = dd.tensors["bp_token"].cpu().numpy()[:IT]
    bp_score = dd.tensors["bp_score"].cpu().numpy()[:IT]
    same_top = 0
    same_trace = 0
    for i, b in enumerate(utts):
        n = int(ref["len"][i])
        top_ok = lens[b] == n and (tokens[b, :n] == ref["tokens"][i, :n]).all()
        same_top += bool(top_ok)
        if top_ok:
            assert abs(scores[b] - ref["score"][i]) <= 1e-3
        # whole trajectory: every iteration's beam (parent, token) and scores
        tr_ok = True
        for it in range(IT):
            ns = int(ref["n_slots"][i, it])
            gp, gt = bp_parent[it, b], bp_token[it, b]
            if (gp >= 0).sum() != ns or (gp[:ns] != ref["parent"][i, it, :ns]).any() or \
                    (gt[:ns] != ref["token"][i, it, :ns]).any():
                tr_ok = False
                break
            if ns:
                assert np.abs(bp_score[it, b, :ns] - ref["tscore"][i, it, :ns]).max() <= 1e-3
        same_trace += tr_ok
    frac = same_top / len(utts)
    assert frac >= min_same, f"top hypothesis identical on {frac:.3f} of utterances"
    return frac, same_trace / len(utts)


def test_search_tiny_unpruned_equals_oracle(Bd):
    # V=32, beam 16 over a tiny net: exercises merging, finished list, empty beams
    dw = synth.decoder(seed=31, V=32, E=32, Hp=32, D=32, Hs=32, Ht=32, tgt_layers=2, U_max=3, W=16)
    e = synth.Stream(4).normal("e", (4, 5, 32)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(5)), 4, 3, 16, min_same=1.0)
    assert tr == 1.0
    fin_n = dd.tensors["fin_n"].cpu().numpy()
    np.testing.assert_array_equal(fin_n, ref["finals_n"])
    fs = dd.tensors["fin_score"].cpu().numpy()
    for b in range(5):
        if fin_n[b]:
            assert np.abs(fs[b, :fin_n[b]] - ref["finals_score"][b, :fin_n[b]]).max() <= 1e-3


@pytest.mark.parametrize("W", [1, 4, 16])
def test_search_beam_widths(Bd, W):
    dw = synth.decoder(seed=41, V=64, E=32, Hp=64, D=32, Hs=32, Ht=64, tgt_layers=2, U_max=8, W=W)
    e = synth.Stream(5).normal("e", (16, 8, 32)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    compare_search(dd, tokens, lens, scores, ref, list(range(8)), 16, 8, W, min_same=1.0)


def test_search_parity_suite_256_utterances(Bd):
    # reduced-dimension end-to-end suite: encoder on the GPU, then the fused search; the
    # top hypothesis must be identical on >= 99 % of the utterances.
    enc_w, dw = synth.parity_suite()
    T, B = enc_w["T"], enc_w["B"]
    got_enc = Bd.Encoder(enc_w["enc"]).forward(torch.from_numpy(enc_w["features"]).cuda())
    e_ref = O.encoder_forward(enc_w["enc"], enc_w["features"])["e"]
    np.testing.assert_array_equal(got_enc["e"].cpu().numpy(), e_ref)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e_ref)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(B)), T, dw.U_max, dw.W)
    print(f"parity suite: top identical {frac:.4f}, whole trajectory identical {tr:.4f}")
    assert tr >= 0.95


def config3_inputs(Bd, T, B):
    act = O.act_symmetric(1.0, 4)
    frames = synth.enc_frames(3, T, B, 1280)
    proj = synth._linear(synth.Stream(3), "enc.proj", 256, 1280)
    fq = Bd.quantize_pack_int4(torch.from_numpy(frames).cuda().reshape(T * B, 1280), to_act(act))
    return Bd.q4_linear_forward(fq, to_act(act), Bd.DeviceLinear(proj)).reshape(T, B, 256)


def test_config3_full_size_sampled_utterances(Bd):
    # beam 16, 16 utterances, target LM 2x2048, source LM 1024, vocabulary 1024: the launch
    # shapes of the full workload (256 hypothesis rows).  The oracle decodes 2 of the 16
    # utterances over the first 24 frames with a label budget of 8 (about a minute of CPU);
    # the GPU runs exactly that setting on all 16.
    dw = synth.decoder(seed=3, U_max=8)
    T, B = 24, 16
    e = config3_inputs(Bd, 300, B)[:T].contiguous().cpu().numpy()
    utts = [1, 14]
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e, utts=utts)
    compare_search(dd, tokens, lens, scores, ref, utts, T, 8, 16, min_same=1.0)


def test_full_size_batch_of_64_sampled_utterance(Bd):
    # 64 utterances x 16 slots = 1024 hypothesis rows at the full layer widths (the batch of the
    # end-to-end workload): 512 tiles per target-LM layer, several per SM.  The oracle decodes
    # one utterance (12 frames, label budget 6).
    dw = synth.decoder(seed=3, U_max=6)
    T, B = 12, 64
    e = config3_inputs(Bd, 12, B).contiguous().cpu().numpy()
    utts = [37]
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e, utts=utts)
    compare_search(dd, tokens, lens, scores, ref, utts, T, 6, 16, min_same=1.0)


def test_tensor_core_and_dp4a_search_paths_agree(Bd):
    # 8 utterances x 16 slots = 128 rows: enough for the tensor-core path; both paths must give
    # identical beams (same integer accumulators, same fp32 operation sequence).
    dw = synth.decoder(seed=51, V=64, E=32, Hp=128, D=32, Hs=128, Ht=256, tgt_layers=2, U_max=10, W=16)
    e = synth.Stream(6).normal("e", (20, 8, 32)).astype(np.float32)
    a = run_search(Bd, dw, e, tensor_cores=True)
    b = run_search(Bd, dw, e, tensor_cores=False)
    for k in ("bp_parent", "bp_token", "fin_n"):
        assert torch.equal(a[0].tensors[k][:30], b[0].tensors[k][:30]), k
    for k in ("bp_score", "fin_score"):       # log-softmax summation order differs between the paths
        x, y = a[0].tensors[k][:30], b[0].tensors[k][:30]
        fin = torch.isfinite(x) & torch.isfinite(y)
        assert torch.equal(torch.isfinite(x), torch.isfinite(y)) and (x[fin] - y[fin]).abs().max().item() <= 1e-3, k
    compare_search(a[0], a[1], a[2], a[3], a[4], list(range(8)), 20, 10, 16, min_same=1.0)


def test_fused_lm_head_small_search(Bd):
    # bottleneck width 256 selects the fused LM-head kernel; 8 utterances x 16 slots, ragged V
    for V in (64, 992):
        dw = synth.decoder(seed=61, V=V, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=6, W=16)
        e = synth.Stream(8).normal("e", (10, 8, 256)).astype(np.float32)
        dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
        compare_search(dd, tokens, lens, scores, ref, list(range(8)), 10, 6, 16, min_same=1.0)
        # the cached LM log-probabilities of live rows are normalised
        rows = dd.tensors["row"].cpu().numpy()
        lp = dd.tensors["tgt_lp"].cpu().numpy()[rows[rows >= 0]]
        if len(lp):
            np.testing.assert_allclose(np.exp(lp.astype(np.float64)).sum(1), 1.0, atol=1e-5)


@pytest.mark.parametrize("V,D", [(46, 256), (37, 64), (300, 256), (1100, 256)])
def test_tensor_core_search_odd_vocabulary(Bd, V, D):
    # the paper's 46 characters and 10-wide embedding (rows of 46 floats are 8-byte aligned only), an odd count
    # without the fused head, and the head's and the selection's other widths (64 columns per CTA; 256, and more
    # labels than a warp holds); 3 utterances x 16 slots, every beam of every iteration
    dw = synth.decoder(seed=63, V=V, E=10, Hp=128, D=D, Hs=128, Ht=256, tgt_layers=2, U_max=6, W=16, out_bits=8)
    e = synth.Stream(18).normal("e", (10, 3, D)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(3)), 10, 6, 16, min_same=1.0)
    assert tr == 1.0


@pytest.mark.parametrize("W,V", [(1, 28940), (2, 19296), (4, 11579), (8, 6400), (12, 4266), (16, 3200), (1, 51200)])
@pytest.mark.parametrize("S,H", [(None, 128), (1, 32)])
def test_search_of_the_largest_vocabularies(Bd, W, V, S, H):
    # the widest vocabularies that the selection's shared memory held once, and the last one that the argument check
    # (200 KB for W x V) lets pass: every beam of every iteration as the oracle's
    dw = synth.decoder(seed=65, V=V, E=32, Hp=H, D=32, Hs=H, Ht=H, tgt_layers=1, U_max=4, W=W)
    e = synth.Stream(W + V).normal("e", (5, 2, 32)).astype(np.float32)
    if S is None:
        dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
        frac, tr = compare_search(dd, tokens, lens, scores, ref, [0, 1], 5, 4, W, min_same=1.0)
    else:
        dd, tokens, lens, scores, ref = run_tsd(Bd, dw, e, S)
        tr = compare_tsd(dd, tokens, lens, scores, ref, [0, 1], 5, S, W)
    assert tr == 1.0
    dw = synth.decoder(seed=65, V=200 * 256 // W + 1, E=32, Hp=32, D=32, Hs=32, Ht=32, tgt_layers=1, U_max=4, W=W)
    with pytest.raises(Bd.Q4Error):
        Bd.Decoder(dw).decode(torch.from_numpy(e).cuda())


def test_search_without_frames(Bd):
    # no frames and, in the alignment-length search, no label budget: no steps, every utterance's string is empty
    dw = synth.decoder(seed=64, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=5, W=8)
    dd = Bd.Decoder(dw)
    e = torch.empty((0, 3, 256), device="cuda")
    for result in (dd.decode(e, u_max=0), dd.decode_time_synchronous(e, 2), dd.decode_time_synchronous(e, 0, u_max=0)):
        tokens, lens, scores = result
        assert lens.tolist() == [0, 0, 0] and scores.tolist() == [0.0, 0.0, 0.0] and not tokens.any()
    with pytest.raises(Bd.Q4Error):
        dd.decode(e, u_max=1)          # a label needs a frame


def test_search_with_cell_states_at_odd_addresses(Bd):
    # cell states that start at no 16-byte boundary: the kernels for unprepared weights take such a search
    dw = synth.decoder(seed=64, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=5, W=8)
    e = synth.Stream(18).normal("e", (12, 3, 256)).astype(np.float32)
    dd = Bd.Decoder(dw)
    dd.alloc_state(3, 8, 17)
    keep = []

    def odd(name):
        n = dd.tensors[name].numel()
        keep.append(torch.zeros(n + 1, device="cuda"))
        return keep[-1][1:].data_ptr()

    dd.state.pred_c, dd.state.src_c = odd("pred_c"), odd("src_c")
    dd.state.tgt_c[0], dd.state.tgt_c[1] = odd("tgt_c0"), odd("tgt_c1")
    tokens, lens, scores = (t.cpu().numpy() for t in dd.decode(torch.from_numpy(e).cuda()))
    assert dd.tensors["status"].item() == 0
    ref = O.alsd(O.Decoder(dw), e)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(3)), 12, 5, 8, min_same=1.0)
    assert tr == 1.0


@pytest.mark.parametrize("V", [20, 46])
@pytest.mark.parametrize("tensor_cores", [True, False])
def test_search_label_budget_of_one(Bd, V, tensor_cores):
    # with a budget of one label the only slot that proposes labels is the empty string, and nearly all of its
    # proposals merge into the blanks of the other slots: too few are left to bound the selection from below
    dw = synth.decoder(seed=65, V=V, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=1, W=16)
    e = synth.Stream(19).normal("e", (12, 6, 256)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e, tensor_cores=tensor_cores)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(6)), 12, 1, 16, min_same=1.0)
    assert tr == 1.0


def test_selection_paths_and_launch_modes_agree(Bd):
    # the bounded fast filter against the exact threshold search, and programmatic dependent
    # launches against plain stream order: bit-identical beams and scores
    dw = synth.decoder(seed=71, V=1024, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=8, W=16)
    e = synth.Stream(9).normal("e", (12, 8, 256)).astype(np.float32)
    base = run_search(Bd, dw, e)
    compare_search(base[0], base[1], base[2], base[3], base[4], list(range(8)), 12, 8, 16, min_same=1.0)
    runs = []
    prev = Bd.beam_select_exact_set(True)
    try:
        runs.append(run_search(Bd, dw, e))
    finally:
        Bd.beam_select_exact_set(prev)
    prev = Bd.dependent_launch_set(False)
    try:
        runs.append(run_search(Bd, dw, e))
    finally:
        Bd.dependent_launch_set(prev)
    for other in runs:
        for k in ("bp_parent", "bp_token", "bp_score", "fin_n", "fin_score", "fin_iter", "fin_slot"):
            assert torch.equal(base[0].tensors[k][:20], other[0].tensors[k][:20]), k
        np.testing.assert_array_equal(base[1], other[1])
        np.testing.assert_array_equal(base[3], other[3])


@pytest.mark.parametrize("V,act_bits", [(1024, 4), (46, 8)])
def test_search_on_one_stream_without_labels(Bd, V, act_bits):
    # 64 rows without side streams; the label budgets are spent early, so that in most iterations every tile of the
    # networks' kernels leaves at once, between the joint network and the selection: the same beams as in plain
    # stream order
    dw = synth.decoder(seed=66, V=V, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=5, W=16, all_bits=act_bits)
    dw.joint.out.bias[0] -= np.float32(10.0)
    e = torch.from_numpy(synth.Stream(22).normal("e", (60, 4, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw, concurrent=False)
    keys = ("bp_parent", "bp_token", "bp_score", "fin_score", "fin_iter", "fin_slot")
    prev = Bd.dependent_launch_set(False)
    try:
        dd.decode(e)
        want = {k: dd.tensors[k].clone() for k in keys}
    finally:
        Bd.dependent_launch_set(prev)
    assert int(((want["bp_token"] > 0).flatten(1).sum(1) == 0).sum()) > 40
    for _ in range(5):
        dd.decode(e)
        for k in keys:
            assert torch.equal(dd.tensors[k], want[k]), k


def check_search_invariants(dd, tokens, lens, scores, T, B, W, U, V=1024):
    """Properties of an alignment-length synchronous search that hold at any size."""
    assert dd.tensors["status"].item() == 0
    IT = T + U
    par = dd.tensors["bp_parent"].cpu().numpy()[:IT]
    tok = dd.tensors["bp_token"].cpu().numpy()[:IT]
    sc = dd.tensors["bp_score"].cpu().numpy()[:IT]
    for b in range(B):
        t = np.zeros(1, np.int64)
        u = np.zeros(1, np.int64)
        strings = [()]
        for it in range(IT):
            n = int((par[it, b] >= 0).sum())
            assert (par[it, b, :n] >= 0).all() and (par[it, b, n:] < 0).all()     # slots are packed
            assert (np.diff(sc[it, b, :n]) <= 0).all()                            # rank order
            p, k = par[it, b, :n], tok[it, b, :n]
            assert (p < len(strings)).all() and (k >= 0).all() and (k < V).all()
            t, u = t[p] + (k == 0), u[p] + (k > 0)
            assert ((t + u) == it + 1).all() and (t < T).all() and (u <= U).all()
            strings = [strings[pp] + ((int(kk),) if kk > 0 else ()) for pp, kk in zip(p, k)]
            assert len(set(strings)) == n                                         # merged: distinct
    fin_n = dd.tensors["fin_n"].cpu().numpy()
    fs = dd.tensors["fin_score"].cpu().numpy()
    lens_h, tok_h, sc_h = lens.cpu().numpy(), tokens.cpu().numpy(), scores.cpu().numpy()
    for b in range(B):
        assert 1 <= fin_n[b] <= W
        assert (np.diff(fs[b, :fin_n[b]]) <= 0).all()
        assert sc_h[b] == fs[b, 0] and 0 <= lens_h[b] <= U
        assert (tok_h[b, :lens_h[b]] > 0).all() and (tok_h[b, lens_h[b]:] == 0).all()


def test_config3_full_length_invariants(Bd):
    # T=300, U_max=150 (450 iterations): properties that hold at any size.
    dw = synth.decoder(seed=3, U_max=150)
    T, B, W, U = 300, 16, 16, 150
    e = config3_inputs(Bd, T, B)
    dd = Bd.Decoder(dw)
    tokens, lens, scores = dd.decode(e)
    torch.cuda.synchronize()
    check_search_invariants(dd, tokens, lens, scores, T, B, W, U)


def test_config4_search_full_size_invariants_in_graph_replay(Bd):
    # The search of the end-to-end workload at its full size and in its launch configuration: 64 utterances,
    # 500 frames, label budget 250 (750 iterations, 1024 hypothesis rows), 8-bit joint output layer, the
    # whole search replayed as one CUDA graph.  Two replays give the same bits, and the properties that hold
    # at any size hold (a search of this length is out of the oracle's reach; its first iterations are
    # covered on sampled utterances by the composed test above).
    dw = synth.decoder(seed=3, out_bits=8, U_max=250)
    T, B, W, U = 500, 64, 16, 250
    e = config3_inputs(Bd, T, B)
    dd = Bd.Decoder(dw)
    run = Bd.GraphedStep(lambda: dd.decode(e))
    t1, l1, s1 = [x.clone() for x in run()]
    par1 = dd.tensors["bp_parent"].clone()
    t2, l2, s2 = run()
    torch.cuda.synchronize()
    assert torch.equal(t1, t2) and torch.equal(l1, l2) and torch.equal(s1, s2)
    assert torch.equal(par1, dd.tensors["bp_parent"])
    check_search_invariants(dd, t2, l2, s2, T, B, W, U)


def run_tsd(Bd, dw, e, S_max, utts=None, tensor_cores=True):
    dd = Bd.Decoder(dw, tensor_cores=tensor_cores)
    tokens, lens, scores = dd.decode_time_synchronous(torch.from_numpy(e).cuda(), S_max)
    torch.cuda.synchronize()
    assert dd.tensors["status"].item() == 0
    ref = O.tsd(O.Decoder(dw), e, S_max, utts=utts)
    return dd, tokens.cpu().numpy(), lens.cpu().numpy(), scores.cpu().numpy(), ref


def compare_tsd(dd, tokens, lens, scores, ref, utts, T, S_max, W):
    IT = T * (S_max + 1)
    bp_parent = dd.tensors["bp_parent"].cpu().numpy()[:IT]
    bp_token = dd.tensors["bp_token"].cpu().numpy()[:IT]
    bp_score = dd.tensors["bp_score"].cpu().numpy()[:IT]
    same = 0
    for i, b in enumerate(utts):
        n = int(ref["len"][i])
        assert lens[b] == n and (tokens[b, :n] == ref["tokens"][i, :n]).all(), (b, tokens[b], ref["tokens"][i])
        assert abs(scores[b] - ref["score"][i]) <= 1e-3
        ok = True
        for it in range(IT):
            ns = int(ref["n_slots"][i, it])
            gp, gt = bp_parent[it, b], bp_token[it, b]
            if (gp >= 0).sum() != ns or (gp[:ns] != ref["parent"][i, it, :ns]).any() or \
                    (gt[:ns] != ref["token"][i, it, :ns]).any():
                ok = False
                break
            if ns:
                assert np.abs(bp_score[it, b, :ns] - ref["tscore"][i, it, :ns]).max() <= 1e-3
        same += ok
    return same / len(utts)


@pytest.mark.parametrize("S_max,W", [(0, 4), (1, 16), (2, 16), (3, 5)])
def test_time_synchronous_search_small(Bd, S_max, W):
    # every set of every call (parents, tokens, provenance of the frame-closing entries) as the oracle's
    dw = synth.decoder(seed=81, V=64, E=32, Hp=64, D=32, Hs=32, Ht=64, tgt_layers=2, U_max=7, W=W)
    e = synth.Stream(12).normal("e", (10, 6, 32)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_tsd(Bd, dw, e, S_max)
    assert compare_tsd(dd, tokens, lens, scores, ref, list(range(6)), 10, S_max, W) == 1.0


@pytest.mark.parametrize("S", [None, 0, 1, 2, 3])
def test_replayed_search_equals_its_steps(Bd, S):
    # searches on one state, long, short, long with other frames (the same graph serves them), then another batch
    # size (built anew): bit-identical to the steps called one by one
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    a, b = Bd.Decoder(dw), Bd.Decoder(dw)
    for B, T, U in ((3, 111, 9), (3, 97, 5), (3, 111, 9), (5, 98, 0)):
        e = torch.from_numpy(synth.Stream(T + B + U).normal("e", (T, B, 256)).astype(np.float32)).cuda()
        n = T + U if S is None else T * (S + 1)
        got = a.decode(e, U) if S is None else a.decode_time_synchronous(e, S, U)
        b.alloc_state(B, 6, n, S)
        b.q4_beam_init()
        for it in range(n):
            b.dr_fusion_beam_step(e, T, it, U, mode=0 if S is None else 2 if it % (S + 1) == S else 1)
        want = b.q4_traceback(n, U)
        for x, y in zip(got, want):
            assert torch.equal(x, y)
        assert a.tensors["status"].item() == 0 and torch.equal(a.tensors["fin_n"], b.tensors["fin_n"])
        for k in ("bp_parent", "bp_token", "bp_score"):
            assert torch.equal(a.tensors[k][:n], b.tensors[k]), k


def test_step_after_a_kernel_that_writes_the_output_scales(Bd):
    # the first call of a frame runs the joint network only; the kernel before it, which lets its successor start
    # early, writes the blank's row scale of the output layer
    dw = synth.decoder(seed=69, V=300, E=32, Hp=128, D=256, Hs=128, Ht=128, U_max=4, W=4)
    e = torch.from_numpy(synth.Stream(21).normal("e", (3, 2, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw)
    write = written_late(Bd, dd.joint_out.w.scale)

    def scores(late):
        dd.alloc_state(2, 4, 6, 1)
        write()
        torch.cuda.synchronize()
        dd.q4_beam_init()
        for it in range(3):
            if late and it == 2:
                write()
            dd.dr_fusion_beam_step(e, 3, it, 4, mode=1 + it % 2)
        torch.cuda.synchronize()
        return torch.cat([dd.tensors["bp_score"][:3].flatten(), dd.tensors["nb_score"].flatten()])

    want = scores(False)
    for _ in range(3):
        assert torch.equal(scores(True), want)


def test_search_plan_builds_and_replays(Bd):
    # groups of 12 steps after the first two frames' steps; one graph serves the searches on a state, another batch
    # size takes another; none below 96 steps, in a capture, or without side streams
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    frames = lambda T, B: torch.from_numpy(synth.Stream(T + B).normal("e", (T, B, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw)
    dd.decode(frames(80, 3), 15)
    assert dd.search_plan_info() == dict(built=0, replays=0, failed=0)     # 95 steps
    dd.alloc_state(3, 6, 120)
    replays = 0
    for T, U in ((81, 15), (111, 9), (97, 5)):
        dd.decode(frames(T, 3), U)
        replays += (T + U - 2) // 12
        assert dd.search_plan_info() == dict(built=1, replays=replays, failed=0)
    dd.decode(frames(111, 5), 9)
    assert dd.search_plan_info() == dict(built=2, replays=replays + 9, failed=0)
    captured = Bd.GraphedStep(lambda e=frames(111, 5): dd.decode(e, 9))
    captured()                                                             # one eager pass, one captured
    assert dd.search_plan_info() == dict(built=2, replays=replays + 18, failed=0)
    plain = Bd.Decoder(dw, concurrent=False)
    plain.decode(frames(111, 5), 9)
    assert plain.search_plan_info() == dict(built=0, replays=0, failed=0)


def test_search_plan_captures_no_stream_of_the_caller(Bd):
    # the side streams lent with the state are not part of the graph: with others in their place it still serves
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    e = torch.from_numpy(synth.Stream(23).normal("e", (111, 3, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw)
    want = [t.clone() for t in dd.decode(e)]
    lent = [torch.cuda.Stream() for _ in range(2)], [torch.cuda.Event() for _ in range(3)]
    for ev in lent[1]:
        ev.record()
    for i in range(2):
        dd.state.aux_stream[i] = lent[0][i].cuda_stream
    for i in range(3):
        dd.state.aux_event[i] = lent[1][i].cuda_event
    for x, y in zip(dd.decode(e), want):
        assert torch.equal(x, y)
    assert dd.search_plan_info() == dict(built=1, replays=18, failed=0)


def test_search_plan_keeps_graphs_of_several_searches(Bd):
    # searches with other fusion weights, in turn on one state: a graph each, up to four, without waiting for the device;
    # with more, the one used longest ago gives way once it has run
    import time
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    e = torch.from_numpy(synth.Stream(24).normal("e", (111, 3, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw)

    def decode(lam):
        dw.lambda_t = lam
        return [t.clone() for t in dd.decode(e)] + [dd.tensors["bp_score"].clone()]

    lams = (0.5, 0.4, 0.3, 0.2, 0.1)
    want = {}
    for lam in lams:
        want[lam] = decode(lam)
        torch.cuda.synchronize()
    assert dd.search_plan_info() == dict(built=5, replays=45, failed=0)
    for _ in range(2):
        for lam in lams[1:]:                     # 0.5 has given way
            for x, y in zip(decode(lam), want[lam]):
                assert torch.equal(x, y)
    assert dd.search_plan_info() == dict(built=5, replays=45 + 72, failed=0)
    torch.cuda.synchronize()
    torch.cuda._sleep(1_000_000_000)             # about half a second
    start = time.perf_counter()
    got = [decode(lam) for lam in (0.1, 0.2, 0.3, 0.4, 0.5)]
    enqueued = time.perf_counter() - start
    torch.cuda.synchronize()
    assert enqueued < 0.5 * (time.perf_counter() - start)
    for g, lam in zip(got, (0.1, 0.2, 0.3, 0.4, 0.5)):
        for x, y in zip(g, want[lam]):
            assert torch.equal(x, y)
    assert dd.search_plan_info()["built"] == 5   # every place was in use: the last search went step by step
    torch.cuda.synchronize()
    decode(0.5)
    assert dd.search_plan_info()["built"] == 6


def test_search_plan_keeps_no_test_hook(Bd):
    # a search while waits of the tiled GEMM are made to run out reports it, and leaves nothing of it in a graph
    import ctypes as C
    dw = synth.decoder(seed=67, V=300, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    e = torch.from_numpy(synth.Stream(25).normal("e", (111, 3, 256)).astype(np.float32)).cuda()
    want = [t.clone() for t in Bd.Decoder(dw).decode(e)]
    dd = Bd.Decoder(dw)
    assert Bd.lib().q4_test_wait_expiry_set(C.c_int32(1), C.c_uint32(1 << 12)) == 0
    try:
        dd.decode(e)
        assert dd.tensors["status"].item() == -8                      # Q4_ERR_TIMEOUT
    finally:
        Bd.lib().q4_test_wait_expiry_set(C.c_int32(0), C.c_uint32(0))
    assert dd.search_plan_info()["replays"] == 0
    for x, y in zip(dd.decode(e), want):
        assert torch.equal(x, y)
    assert dd.tensors["status"].item() == 0


@pytest.mark.parametrize("where", [1, 2])
def test_search_whose_loop_cannot_be_built(Bd, where):
    # the loop's node is refused, or cannot be filled: the steps are enqueued, or captured by the caller, one by one
    import ctypes as C
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    e = torch.from_numpy(synth.Stream(26).normal("e", (111, 3, 256)).astype(np.float32)).cuda()
    plain = Bd.Decoder(dw, concurrent=False)
    want = [t.clone() for t in plain.decode(e)]
    dd = Bd.Decoder(dw)
    dd.alloc_state(3, 6, 120)
    dd.decode(e[:30], 5)                                                   # short: makes the plan, builds nothing
    fail = lambda x: Bd.lib().q4_test_search_loop_failure_set(dd._plan.handle, C.c_int32(x))
    captured = Bd.GraphedStep(lambda: dd.decode(e))
    assert fail(3) != 0 and fail(where) == 0
    for run in (lambda: dd.decode(e), captured, captured):                 # (the second makes an eager pass and a captured one)
        dd.tensors["bp_score"].fill_(-7)
        for x, y in zip(run(), want):
            assert torch.equal(x, y)
        assert dd.tensors["status"].item() == 0 and torch.equal(dd.tensors["bp_score"], plain.tensors["bp_score"])
    assert dd.search_plan_info() == dict(built=0, replays=0, failed=3)
    assert fail(0) == 0
    looped = Bd.GraphedStep(lambda: dd.decode(e))
    for run in (looped, looped):
        for x, y in zip(run(), want):
            assert torch.equal(x, y)
    assert dd.search_plan_info() == dict(built=1, replays=9, failed=3)


@pytest.mark.parametrize("W,H", [(6, 256), (16, 1024)])
def test_products_stay_until_their_copies_have_landed(Bd, W, H):
    # Waits of the recurrent sums' kernel give up at once, or after one poll, while its copies are on their way, fewer and more
    # of them than its ring holds: a search has the right scores or reads Q4_ERR_TIMEOUT, and the next one is right.
    import ctypes as C
    dw = synth.decoder(seed=67, V=64, E=32, Hp=H, D=256, Hs=H, Ht=H, tgt_layers=2, U_max=9, W=W)
    e = torch.from_numpy(synth.Stream(29).normal("e", (20, 3, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw)
    want = [t.clone() for t in dd.decode(e)] + [dd.tensors["bp_score"].clone()]
    for limit in (0, 0, 1, 0):
        assert Bd.lib().q4_test_wait_expiry_set(C.c_int32(2), C.c_uint32(limit)) == 0
        try:
            got = dd.decode(e)
            torch.cuda.synchronize()
        finally:
            Bd.lib().q4_test_wait_expiry_set(C.c_int32(0), C.c_uint32(0))
        status = dd.tensors["status"].item()
        assert status == -8 or (limit and status == 0 and torch.equal(dd.tensors["bp_score"], want[3]))   # Q4_ERR_TIMEOUT
        for x, y in zip([*dd.decode(e), dd.tensors["bp_score"]], want):
            assert torch.equal(x, y)
        assert dd.tensors["status"].item() == 0


def test_search_beside_a_capture_of_another_thread(Bd):
    # a search that creates its plan and builds its graph on one thread leaves a capture that another thread has open
    # (in the strictest mode, torch's default) as it is
    import threading
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    e = torch.from_numpy(synth.Stream(23).normal("e", (111, 3, 256)).astype(np.float32)).cuda()
    first = Bd.Decoder(dw)
    first.decode(e)                          # kernels are loaded
    dd = Bd.Decoder(dw, share_from=first)
    dd.alloc_state(3, 6, 120)
    x = torch.zeros(8, device="cuda")
    side, capturing, failure = torch.cuda.Stream(), torch.cuda.Stream(), []
    while capturing in (side, *dd._aux_streams):         # torch hands its streams out in turn, more than once
        capturing = torch.cuda.Stream()

    def search():
        try:
            for lam in (dw.lambda_t, 0.25):                  # the second search builds another graph
                dd.dw.lambda_t = lam
                with torch.cuda.stream(side):
                    dd.q4_beam_init()
                    dd.q4_beam_search(e, 111, 9)
        except Exception as error:
            failure.append(error)

    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=capturing):
        x.add_(1.0)
        worker = threading.Thread(target=search)
        worker.start()
        worker.join()
        x.add_(2.0)
    assert not failure, failure
    x.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [3.0] * 8
    assert dd.search_plan_info() == dict(built=2, replays=18, failed=0)


def test_time_synchronous_search_tensor_core_path(Bd):
    # 8 utterances x 16 slots = 128 rows and a 256-wide bottleneck: tensor-core LSTMs and cluster heads
    dw = synth.decoder(seed=83, V=128, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=16)
    e = synth.Stream(13).normal("e", (8, 8, 256)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_tsd(Bd, dw, e, 2)
    assert compare_tsd(dd, tokens, lens, scores, ref, list(range(8)), 8, 2, 16) == 1.0
    # the alignment-length synchronous search still runs on a decoder that has just done this one
    t2, l2, s2 = dd.decode(torch.from_numpy(e).cuda())
    r2 = O.alsd(O.Decoder(dw), e, trace=False)
    for b in range(8):
        n = int(r2["len"][b])
        assert l2[b].item() == n and (t2[b, :n].cpu().numpy() == r2["tokens"][b, :n]).all()


def test_config3_time_synchronous_full_size_sampled_utterances(Bd):
    # the beam workload's sizes (target LM 2x2048, source LM 1024, vocabulary 1024, 16 utterances x 16
    # slots), 8 frames x 3 calls, label budget 8; the oracle decodes 2 of the 16 utterances
    dw = synth.decoder(seed=3, U_max=8)
    T, B = 8, 16
    e = config3_inputs(Bd, 300, B)[:T].contiguous().cpu().numpy()
    utts = [2, 13]
    dd, tokens, lens, scores, ref = run_tsd(Bd, dw, e, 2, utts=utts)
    assert compare_tsd(dd, tokens, lens, scores, ref, utts, T, 2, 16) == 1.0


def test_time_synchronous_mode_checks(Bd):
    dw = synth.decoder(seed=81, V=64, E=32, Hp=64, D=32, Hs=32, Ht=64, tgt_layers=2, U_max=4, W=4)
    dd = Bd.Decoder(dw)
    e = torch.zeros((3, 2, 32), device="cuda")
    dd.alloc_state(2, 4, 9)                      # layout of the alignment-length synchronous search
    dd.q4_beam_init()
    with pytest.raises(RuntimeError):            # no candidate set in this state
        dd.dr_fusion_beam_step(e, 3, 0, 4, mode=1)
    dd.alloc_state(2, 4, 9, S_max=2)
    dd.q4_beam_init()
    with pytest.raises(RuntimeError):            # call 0 of a frame is not the closing one
        dd.dr_fusion_beam_step(e, 3, 0, 4, mode=2)
    with pytest.raises(RuntimeError):            # beyond the last frame
        dd.dr_fusion_beam_step(e, 3, 9, 4, mode=1)


# ------------------------------------------------------------------ gaps closed after review
def beam_strings(dd, n_iters, B):
    """Label string of every slot of the beam after n_iters iterations, from the history."""
    par = dd.tensors["bp_parent"].cpu().numpy()[:n_iters]
    tok = dd.tensors["bp_token"].cpu().numpy()[:n_iters]
    out = []
    for b in range(B):
        strings = [()]
        for it in range(n_iters):
            n = int((par[it, b] >= 0).sum())
            strings = [strings[p] + ((int(k),) if k > 0 else ()) for p, k in zip(par[it, b, :n], tok[it, b, :n])]
        out.append(strings)
    return out


@pytest.mark.parametrize("V", [1024, 992])
def test_lm_logprobs_elementwise_through_the_search(Bd, V):
    # The LM rows the search caches (LSTM layers -> bottleneck -> re-quantize -> output -> log-softmax,
    # the fused head kernel) against the oracle's forced LM on each live hypothesis' label string,
    # element by element; also the joint's projected prediction vectors.  9 utterances x 16 slots.
    dw = synth.decoder(seed=91, V=V, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=6, W=16)
    B, T, n_it = 9, 8, 7
    e = synth.Stream(14).normal("e", (T, B, 256)).astype(np.float32)
    dd = Bd.Decoder(dw)
    dd.alloc_state(B, 16, T + 6)
    dd.q4_beam_init()
    e_dev = torch.from_numpy(e).cuda()
    for it in range(n_it):
        dd.dr_fusion_beam_step(e_dev, T, it, 6)
    torch.cuda.synchronize()
    strings = beam_strings(dd, n_it, B)
    dec = O.Decoder(dw)
    # a slot without a pending advance stands on a state row whose networks have been run
    rows = dd.tensors["row"].cpu().numpy().reshape(B, 16)
    adv_dst = dd.tensors["adv_dst"].cpu().numpy().reshape(B, 16)
    tgt_lp = dd.tensors["tgt_lp"].cpu().numpy()
    src_lp = dd.tensors["src_lp"].cpu().numpy()
    pred_p = dd.tensors["pred_p"].cpu().numpy()
    n_rows = worst = 0
    for b in range(B):
        for s, y in enumerate(strings[b]):
            r = rows[b, s]
            if r < 0 or adv_dst[b, s] >= 0:
                continue
            toks = np.array([[0] + list(y)], dtype=np.int32)
            for which, lp in (("tgt", tgt_lp), ("src", src_lp)):
                want = O.lm_forced(dec, which, toks)[0, -1]
                err = np.abs(lp[r] - want).max()
                worst = max(worst, err)
                assert err <= LP_ATOL, (b, s, which, err)
            fi = np.zeros((1, toks.shape[1]), np.int32)
            _, _, _, p_w = O.pred_joint_forced(dec, e[:, b], fi, toks, want_state=True)
            np.testing.assert_array_equal(pred_p[r], p_w[0, -1])
            n_rows += 1
    print(f"V={V}: {n_rows} cached LM rows compared element-wise, worst |d log P| = {worst:.2e}")
    assert n_rows >= 100


@pytest.mark.parametrize("W", [1, 16])
def test_single_utterance_full_widths(Bd, W):
    # ONE utterance at the full layer widths (the regime of the paper's run-time figure, Section 4.1):
    # at most 16 hypothesis rows in one padded row tile, all three chains on the small-call stream plan
    dw = synth.decoder(seed=3, U_max=6, W=W)
    T = 12
    e = config3_inputs(Bd, T, 1).contiguous().cpu().numpy()
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, [0], T, 6, W, min_same=1.0)
    assert tr == 1.0


def test_single_utterance_full_length_beam_4(Bd):
    # the run-time figure's utterance at its full length (152 frames, label budget 76: 228 iterations) and
    # full widths, beam 4 (what the oracle decodes in a fraction of a minute): every beam of every iteration
    # identical, through both regimes of the search (label iterations, then label-free ones)
    dw = synth.decoder(seed=3, U_max=76, W=4)
    T = 152
    e = config3_inputs(Bd, T, 1).contiguous().cpu().numpy()
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, [0], T, 76, 4, min_same=1.0)
    assert tr == 1.0


def test_config4_composed_full_widths_sampled_utterances(Bd):
    # The end-to-end workload as composed, at full widths and with its batch of 64: log-mel ->
    # prologue -> per-utterance MAX boundary, 8-bit first encoder layer -> 4-bit layers 2-6 ->
    # projection -> beam-16 fused search with the 8-bit joint output layer.  24 log-mel frames
    # (12 encoder frames), label budget 6; the oracle runs two of the 64 utterances.
    B, T100, U = 64, 24, 6
    T = T100 // 2
    enc_w = synth.encoder(4, T=T, B=B, first_layer_bits=8, in_max=True, features=False)
    dw = synth.decoder(3, out_bits=8, U_max=U)
    mel = synth.logmel(4, B, T100, 40)
    feats_dev = Bd.q4_feature_prologue(torch.from_numpy(mel).cuda())
    enc = Bd.Encoder(enc_w["enc"])
    got = enc.forward(feats_dev, want_layers=True)
    utts = [5, 58]
    feats_ref = np.stack([O.features(mel[b]) for b in utts], axis=1).astype(np.float16)
    np.testing.assert_array_equal(feats_dev.cpu().numpy()[:, utts], feats_ref)
    ref_enc = O.encoder_forward(enc_w["enc"], feats_ref, want_layers=True)
    for l, yq in enumerate(got["layers"]):
        g = gpu_codes(yq, 1280, enc.out_acts[l]).reshape(T, B, 1280)[:, utts]
        np.testing.assert_array_equal(g, ref_enc["layers"][l]["yq"], err_msg=f"encoder layer {l}")
    e_gpu = got["e"].cpu().numpy()
    np.testing.assert_array_equal(e_gpu[:, utts], ref_enc["e"])
    dd = Bd.Decoder(dw)
    tokens, lens, scores = dd.decode(got["e"])
    torch.cuda.synchronize()
    assert dd.tensors["status"].item() == 0
    ref = O.alsd(O.Decoder(dw), ref_enc["e"])
    frac, tr = compare_search(dd, tokens.cpu().numpy(), lens.cpu().numpy(), scores.cpu().numpy(), ref,
                              utts, T, U, 16, min_same=1.0)
    assert tr == 1.0


@pytest.mark.parametrize("tensor_cores", [True, False])
def test_search_two_bit_rnnt_weights(Bd, tensor_cores):
    # Table 1's 2/4 rows: prediction and joint network weights stored at 2 bits under 4-bit
    # activations, LMs at 4 bits; 8 utterances x 16 slots, every beam of every iteration
    dw = synth.decoder(seed=95, V=64, E=64, Hp=128, D=64, Hs=128, Ht=128, tgt_layers=2, U_max=6, W=16,
                       rnnt_w_bits=2)
    assert dw.pred.lstm.w_ih.bits == 2 and dw.joint.out.w.bits == 2 and dw.tgt.lstm[0].w_ih.bits == 4
    e = synth.Stream(15).normal("e", (10, 8, 64)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e, tensor_cores=tensor_cores)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(8)), 10, 6, 16, min_same=1.0)
    assert tr == 1.0


@pytest.mark.parametrize("dims", [dict(V=64, E=32, Hp=64, D=32, Hs=32, Ht=64), dict(V=128, E=32, Hp=128, D=256, Hs=128, Ht=256)])
def test_search_all_eight_bit(Bd, dims):
    # every weight and every activation quantizer of the decoder at 8 bits (the all-8-bit point of the
    # paper's run-time figure): 8-bit search state, DP4A kernels (small) and tensor-core kernels
    dw = synth.decoder(seed=97, tgt_layers=2, U_max=6, W=16, all_bits=8, **dims)
    assert dw.pred.lstm.w_hh.bits == 8 and dw.tgt.out.w.bits == 8 and dw.pred.lstm.hid_bits == 8
    e = synth.Stream(16).normal("e", (10, 8, dims["D"])).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    assert dd.tensors["pred_hq"].shape[1] == dims["Hp"]           # one byte per hidden code
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(8)), 10, 6, 16, min_same=1.0)
    assert tr == 1.0


@pytest.mark.parametrize("single_steps", [True, False])
@pytest.mark.parametrize("B,W", [(1, 5), (1, 16), (2, 16), (3, 7)])
def test_search_few_rows_weight_streaming_kernels(Bd, B, W, single_steps):
    # at most 32 hypothesis rows and widths that are multiples of 128: the LSTM steps of single steps run on the
    # weight-streaming kernel that reads packed 4-bit weights, state rows and embedding rows as stored
    # (signed prediction-network input, unsigned LM input with its zero point), those of a whole search on the kernels that
    # look labels up and keep sums; every beam of every iteration as the oracle's
    dw = synth.decoder(seed=99, V=128, E=128, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=6, W=W)
    e = synth.Stream(17).normal("e", (9, B, 256)).astype(np.float32)
    if single_steps:
        dd = Bd.Decoder(dw)
        dd.alloc_state(B, W, 15)
        dd.q4_beam_init()
        e_dev = torch.from_numpy(e).cuda()
        for it in range(15):
            dd.dr_fusion_beam_step(e_dev, 9, it, 6)
        tokens, lens, scores = (t.cpu().numpy() for t in dd.q4_traceback(15, 6))
        assert dd.tensors["status"].item() == 0
        ref = O.alsd(O.Decoder(dw), e)
    else:
        dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(B)), 9, 6, W, min_same=1.0)
    assert tr == 1.0


def test_grouped_search_equals_single_state_search(Bd):
    # the batch searched as two and three sets of utterances side by side (own states and streams, one copy
    # of the weights): token for token, score for score, the result of the one-state search
    dw = synth.decoder(seed=101, V=64, E=32, Hp=128, D=32, Hs=128, Ht=256, tgt_layers=2, U_max=8, W=16)
    e = synth.Stream(18).normal("e", (14, 12, 32)).astype(np.float32)
    e_dev = torch.from_numpy(e).cuda()
    one = Bd.Decoder(dw)
    t1, l1, s1 = one.decode(e_dev)
    torch.cuda.synchronize()
    for G in (2, 3):
        gd = Bd.GroupedDecoder(dw, G)
        t2, l2, s2 = gd.decode(e_dev)
        torch.cuda.synchronize()
        assert torch.equal(t1, t2) and torch.equal(l1, l2) and torch.equal(s1, s2)
        assert torch.equal(gd.history("bp_parent")[:22], one.tensors["bp_parent"][:22])
        assert torch.equal(gd.history("bp_token")[:22], one.tensors["bp_token"][:22])
        # and replayed as a CUDA graph
        g = Bd.GraphedStep(lambda: gd.decode(e_dev))
        t3, l3, s3 = g()
        t3, l3, s3 = g()
        torch.cuda.synchronize()
        assert torch.equal(t1, t3) and torch.equal(s1, s3)


@pytest.mark.parametrize("V,W,B,T,U,blank,bits", [
    (46, 16, 3, 101, 7, 2.0, 4),      # vocabulary summed by a warp per row; utterances that spend their labels at different times
    (256, 5, 2, 130, 30, 0.0, 8),
    (257, 16, 2, 97, 20, 3.0, 4),     # blocks of 64 labels
    (1024, 16, 5, 110, 12, 4.0, 4),   # blocks of 128
    (1000, 1, 1, 300, 0, 0.0, 4),     # no label budget: everything is left to the end; a last block with few labels
    (1030, 8, 2, 100, 90, -9.0, 8),   # blocks of 256; hardly any blank before the labels are spent
    (300, 4, 2, 100, 60, 30.0, 4),    # blanks only: the beams end before any label budget is spent
])
def test_label_free_end_of_a_search_equals_its_steps(Bd, V, W, B, T, U, blank, bits):
    # the iterations after the last label are carried out together: every beam of every iteration, the finished list and
    # the state as the steps leave them, in a search of its own and in one captured by the caller
    dw = synth.decoder(seed=91, V=V, E=32, Hp=128, D=256, Hs=128, Ht=128, tgt_layers=2, U_max=U, W=W, all_bits=bits)
    dw.joint.out.bias[0] += np.float32(blank)
    e = torch.from_numpy(synth.Stream(V + T).normal("e", (T, B, 256)).astype(np.float32)).cuda()
    n = T + U
    b = Bd.Decoder(dw)
    b.alloc_state(B, W, n)
    b.q4_beam_init()
    for it in range(n):
        b.dr_fusion_beam_step(e, T, it, U)
    want = b.q4_traceback(n, U)
    a = Bd.Decoder(dw)
    captured = Bd.GraphedStep(lambda: a.decode(e, U))
    state = ("bp_parent", "bp_token", "bp_score", "fin_n", "fin_score", "fin_iter", "fin_slot", "score", "t", "u", "hash",
             "prev_hash", "last_tok", "row", "adv_src", "adv_dst", "adv_tok", "pend_n")
    for run in (lambda: a.decode(e, U), captured, captured):
        if a.state is not None:
            for k in ("bp_parent", "bp_token", "bp_score"):
                a.tensors[k].fill_(-7)
        got = run()
        assert a.tensors["status"].item() == 0
        for x, y in zip(got, want):
            assert torch.equal(x, y)
        for k in state:
            assert torch.equal(a.tensors[k], b.tensors[k]), k
    assert a.search_plan_info()["built"] == 1


@pytest.mark.parametrize("T,U,S", [(111, 9, None), (100, 12, None), (30, 5, None), (60, 4, 1)])
def test_search_counts_the_quantizers_of_all_its_steps(Bd, T, U, S):
    # prediction, source and two target layers, two bottlenecks and tanh(e p) a step: in a looped, captured, replayed or plain
    # search, whether its steps are a multiple of a graph's or not
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=U, W=6)
    e = torch.from_numpy(synth.Stream(27).normal("e", (T, 3, 256)).astype(np.float32)).cuda()
    n = T + U if S is None else T * (S + 1)
    for concurrent in (True, False):
        dd = Bd.Decoder(dw, concurrent=concurrent)
        run = (lambda: dd.decode(e)) if S is None else (lambda: dd.decode_time_synchronous(e, S))
        run()
        Bd.quantizer_calls(reset=True)
        run()
        assert Bd.quantizer_calls(reset=True) == 7 * n
        Bd.GraphedStep(run)()                                  # an eager pass and a captured one
        assert Bd.quantizer_calls(reset=True) == 14 * n


def test_steps_that_a_search_has_taken(Bd):
    # without labels a loop takes one turn of 12 steps behind the first two; a search that is not looped takes all of its own,
    # whatever ran on the state before
    dw = synth.decoder(seed=67, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=9, W=6)
    e = torch.from_numpy(synth.Stream(28).normal("e", (110, 3, 256)).astype(np.float32)).cuda()
    dd = Bd.Decoder(dw)
    dd.alloc_state(3, 6, 220)
    captured = Bd.GraphedStep(lambda: dd.decode(e, 0))
    for run, low, high in ((lambda: dd.decode(e, 0), 14, 14), (lambda: dd.decode(e[:50], 5), 55, 55), (captured, 14, 14),
                           (lambda: dd.decode(e, 9), 14, 119)):
        run()
        assert low <= dd.search_steps_taken() <= high
    plain = Bd.Decoder(dw, concurrent=False)
    plain.decode(e, 9)
    assert plain.search_steps_taken() == 119
    dd.decode_time_synchronous(e, 1, 9)
    assert dd.search_steps_taken() == 220


@pytest.mark.parametrize("V,normalized", [(2, 1), (46, 1), (64, 1), (65, 1), (256, 1), (257, 1), (300, 0), (1023, 1), (1024, 0),
                                          (1024, 1), (1025, 1)])
@pytest.mark.parametrize("S", [None, 1])
def test_selection_forms_agree_with_the_exact_search(Bd, V, normalized, S):
    # every form of the selection kernels (labels per lane, rows of whole 16 bytes, logits or log-probabilities, more labels
    # than registers hold) against the exact threshold search, with few and many slots
    D = 256 if normalized else 128
    dw = synth.decoder(seed=93, V=V, E=32, Hp=128, D=D, Hs=128, Ht=128, tgt_layers=1, U_max=6, W=16)
    for B, W in ((2, 16), (3, 5), (9, 15)):
        e = torch.from_numpy(synth.Stream(V + W).normal("e", (10, B, D)).astype(np.float32)).cuda()
        runs = []
        for exact in (False, True):
            dd = Bd.Decoder(dw)
            prev = Bd.beam_select_exact_set(exact)
            try:
                out = dd.decode(e, 6, W) if S is None else dd.decode_time_synchronous(e, S, 6, W)
                torch.cuda.synchronize()
            finally:
                Bd.beam_select_exact_set(prev)
            runs.append(list(out) + [dd.tensors[k] for k in ("bp_parent", "bp_token", "bp_score", "fin_n", "fin_score")])
        for x, y in zip(*runs):
            assert torch.equal(x, y)


@pytest.mark.parametrize("V", [260, 516, 1000, 1024])
@pytest.mark.parametrize("S,D,tensor_cores", [(None, 64, True), (1, 64, True), (None, 256, False), (None, 256, True)])
def test_selection_of_rows_at_smaller_alignments(Bd, V, S, D, tensor_cores):
    # logits and log-probabilities, in the form that reads rows 16 bytes at a time and, with a language model's rows at a
    # 4-byte boundary, in the one that reads single elements: the same bits
    dw = synth.decoder(seed=94, V=V, E=32, Hp=128, D=D, Hs=128, Ht=128, tgt_layers=1, U_max=6, W=16)
    for B, W in ((1, 16), (3, 5)):
        e = torch.from_numpy(synth.Stream(V + W).normal("e", (10, B, D)).astype(np.float32)).cuda()
        runs = []
        for shift in (0, 1):
            dd = Bd.Decoder(dw, tensor_cores=tensor_cores)
            dd.alloc_state(B, W, 16 if S is None else 20, S)
            rows = torch.zeros(dd.tensors["src_lp"].numel() + 4, device="cuda")
            dd.state.src_lp = rows[shift:].data_ptr()
            out = dd.decode(e, 6, W) if S is None else dd.decode_time_synchronous(e, S, 6, W)
            runs.append(list(out) + [dd.tensors[k] for k in ("bp_parent", "bp_token", "bp_score", "fin_n", "fin_score", "status")])
        for x, y in zip(*runs):
            assert torch.equal(x, y)


@pytest.mark.parametrize("B,W,S,layers,bits", [(3, 7, None, 2, 4), (8, 16, None, 2, 4), (9, 15, 1, 2, 4), (24, 16, None, 1, 8),
                                               (25, 16, None, 2, 4), (2, 16, 3, 1, 4)])
def test_search_that_keeps_sums_equals_its_steps(Bd, B, W, S, layers, bits):
    # tables for the input halves and recurrent sums per state row against the step kernels: the edges of row tiles, the
    # largest search that keeps them and one more, one or two target-LM layers
    dw = synth.decoder(seed=95, V=300, E=32, Hp=256, D=256, Hs=128, Ht=384, tgt_layers=layers, U_max=12, W=W, all_bits=bits)
    dw.joint.out.bias[0] += np.float32(2.0)
    T = 30
    e = torch.from_numpy(synth.Stream(B + W).normal("e", (T, B, 256)).astype(np.float32)).cuda()
    n = T + 12 if S is None else T * (S + 1)
    a, b = Bd.Decoder(dw), Bd.Decoder(dw)
    got = a.decode(e, 12) if S is None else a.decode_time_synchronous(e, S, 12)
    b.alloc_state(B, W, n, S)
    b.q4_beam_init()
    for it in range(n):
        b.dr_fusion_beam_step(e, T, it, 12, mode=0 if S is None else 2 if it % (S + 1) == S else 1)
    for x, y in zip(got, b.q4_traceback(n, 12)):
        assert torch.equal(x, y)
    assert a.tensors["status"].item() == 0
    for k in ("bp_parent", "bp_token", "bp_score", "fin_n", "fin_score", "pred_c", "tgt_c0", "tgt_hq0", "pred_p"):
        assert torch.equal(a.tensors[k], b.tensors[k]), k


@pytest.mark.parametrize("B,W,S", [(9, 15, None), (16, 16, None), (24, 16, None), (17, 8, 1), (24, 16, 2)])
def test_replayed_search_that_keeps_sums_equals_its_steps(Bd, B, W, S):
    # the same from a graph (a loop, or groups of steps), where the products of one, two and three row tiles have a stream of
    # their own beside the heads and the selection: the decoder's graph twice, and one captured by the caller twice
    dw = synth.decoder(seed=92, V=300, E=32, Hp=256, D=256, Hs=128, Ht=384, tgt_layers=2, U_max=25, W=W)
    dw.joint.out.bias[0] += np.float32(3.0)
    T, U = (101, 25) if S is None else (50, 25)
    e = torch.from_numpy(synth.Stream(B * W).normal("e", (T, B, 256)).astype(np.float32)).cuda()
    n = T + U if S is None else T * (S + 1)
    a, b = Bd.Decoder(dw), Bd.Decoder(dw)
    b.alloc_state(B, W, n, S)
    b.q4_beam_init()
    for it in range(n):
        b.dr_fusion_beam_step(e, T, it, U, mode=0 if S is None else 2 if it % (S + 1) == S else 1)
    want = b.q4_traceback(n, U)
    decode = (lambda: a.decode(e, U)) if S is None else (lambda: a.decode_time_synchronous(e, S, U))
    captured = Bd.GraphedStep(decode)
    keys = ["bp_parent", "bp_token", "bp_score", "fin_n", "fin_score", "fin_iter", "fin_slot", "score", "row", "status", "pred_c",
            "src_c", "tgt_c0", "tgt_c1", "pred_hq", "src_hq", "tgt_hq0", "tgt_hq1", "pred_p", "src_lp", "tgt_lp"]
    for run in (decode, decode, captured, captured):
        if a.state is not None:
            for k in keys[:3] + keys[10:14]:
                a.tensors[k].fill_(0)
        for x, y in zip(run(), want):
            assert torch.equal(x, y)
        for k in keys:
            assert torch.equal(a.tensors[k], b.tensors[k]), k
    assert a.search_plan_info()["built"] == 1 and a.model.tables


def test_search_with_embeddings_of_other_row_lengths(Bd):
    # 2-bit weights of the prediction network pad its 10-wide embedding rows to 64 codes, the language models' to 32: the
    # tables take each network's own, and the beams are the oracle's
    dw = synth.decoder(seed=96, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=5, W=8, rnnt_w_bits=2)
    e = synth.Stream(31).normal("e", (12, 3, 256)).astype(np.float32)
    dd, tokens, lens, scores, ref = run_search(Bd, dw, e)
    assert dd.pred_lstm.w_ih.k_pad != dd.src.lstm[0].w_ih.k_pad
    frac, tr = compare_search(dd, tokens, lens, scores, ref, list(range(3)), 12, 5, 8, min_same=1.0)
    assert tr == 1.0


@pytest.mark.parametrize("what", ["workspace", "prepared", "pred_p"])
def test_search_with_buffers_at_smaller_alignments(Bd, what):
    # a workspace or prepared weights at a 16-byte boundary, projected prediction rows at an 8-byte one: kernels that move more
    # at a time are not taken, the beams are the same
    import ctypes as C
    dw = synth.decoder(seed=97, V=300, E=32, Hp=128, D=256, Hs=128, Ht=128, tgt_layers=2, U_max=9, W=6)
    dw.joint.out.bias[0] += np.float32(3.0)
    e = torch.from_numpy(synth.Stream(33).normal("e", (100, 3, 256)).astype(np.float32)).cuda()
    a, b = Bd.Decoder(dw), Bd.Decoder(dw)
    want = b.decode(e)
    a.alloc_state(3, 6, 109)
    shift = 8 if what == "pred_p" else 16

    def moved(t):
        big = torch.zeros(t.numel() * t.element_size() + 32, dtype=torch.uint8, device="cuda")
        return big[shift:shift + t.numel() * t.element_size()].view(t.dtype).view(t.shape)

    if what == "workspace":
        a.ws = moved(a.ws)
    elif what == "prepared":
        a.prepared = moved(a.prepared)
        assert Bd.lib().q4_prepare_model(C.byref(a.model), C.c_void_p(a.prepared.data_ptr()), C.c_size_t(a.prepared.numel()), None) == 0
        torch.cuda.synchronize()
    else:
        a.tensors["pred_p"] = moved(a.tensors["pred_p"])
        a.state.pred_p = a.tensors["pred_p"].data_ptr()
    got = a.decode(e)
    for x, y in zip(got, want):
        assert torch.equal(x, y)
    assert a.tensors["status"].item() == 0
    for k in ("bp_parent", "bp_token", "bp_score"):
        assert torch.equal(a.tensors[k][:109], b.tensors[k][:109]), k


def test_embeddings_after_the_preparation_of_the_weights(Bd):
    # q4_prepare_model reads no embedding tables: it takes a model without them, and a search follows what they hold when it
    # runs, unless tables have been made from them, which are made again with the weights
    import copy
    import ctypes as C
    dw = synth.decoder(seed=96, V=46, E=10, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=5, W=8)
    other = copy.deepcopy(dw)
    for part in (other.pred, other.src, other.tgt):
        part.emb = -part.emb
    e = torch.from_numpy(synth.Stream(31).normal("e", (12, 3, 256)).astype(np.float32)).cuda()
    a, b = Bd.Decoder(dw), Bd.Decoder(other)
    want = [t.clone() for t in b.decode(e)] + [b.tensors["bp_score"]]
    before = [t.clone() for t in a.decode(e)] + [a.tensors["bp_score"].clone()]
    assert not torch.equal(before[-1], want[-1])

    def check(d):
        for x, y in zip([*d.decode(e), d.tensors["bp_score"]], want):
            assert torch.equal(x, y)

    for x, y in ((a.pred_emb_q, b.pred_emb_q), (a.src.emb_q, b.src.emb_q), (a.tgt.emb_q, b.tgt.emb_q)):
        x.copy_(y)
    a.model.tables = None
    check(a)
    m = Bd.Decoder(dw)
    tables = m.model.pred_emb_q, m.model.src.emb_q, m.model.tgt.emb_q
    m.model.pred_emb_q = m.model.src.emb_q = m.model.tgt.emb_q = None
    m.q4_prepare_model()
    m.model.pred_emb_q, m.model.src.emb_q, m.model.tgt.emb_q = tables
    for x, y in ((m.pred_emb_q, b.pred_emb_q), (m.src.emb_q, b.src.emb_q), (m.tgt.emb_q, b.tgt.emb_q)):
        x.copy_(y)
    check(m)
    assert m.model.tables and not Bd.lib().q4_table_bytes(C.byref(m.model), C.c_int32(385))
    for x in (m.pred_emb_q, m.src.emb_q, m.tgt.emb_q):       # other codes, tables of them, then the codes of before
        x.fill_(0x11)
    m.q4_prepare_model()
    assert not torch.equal(m.decode(e)[2], want[2])
    for x, y in zip((m.pred_emb_q, m.src.emb_q, m.tgt.emb_q), (b.pred_emb_q, b.src.emb_q, b.tgt.emb_q)):
        x.copy_(y)
    m.q4_prepare_model()
    check(m)


def test_tables_made_on_another_stream(Bd):
    # a decoder that shares the weights takes the tables that the first one is still making, late on its own stream
    dw = synth.decoder(seed=96, V=300, E=32, Hp=128, D=256, Hs=128, Ht=256, tgt_layers=2, U_max=5, W=8)
    e = torch.from_numpy(synth.Stream(34).normal("e", (12, 3, 256)).astype(np.float32)).cuda()
    want = [t.clone() for t in Bd.Decoder(dw).decode(e)]
    first = Bd.Decoder(dw)
    second = Bd.Decoder(dw, share_from=first)
    torch.cuda.synchronize()
    late, side = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(late):
        torch.cuda._sleep(200_000_000)                         # a tenth of a second
        first.alloc_state(3, 8, 17)
    with torch.cuda.stream(side):
        got = second.decode(e)
    torch.cuda.synchronize()
    assert first.model.tables and second.tables is first.tables
    for x, y in zip(got, want):
        assert torch.equal(x, y)


def test_search_with_prepared_weights_at_a_16_byte_boundary_and_tables(Bd):
    # tables have a buffer of their own: weights at a 16-byte boundary serve the kernels that look labels up
    import ctypes as C
    dw = synth.decoder(seed=97, V=300, E=32, Hp=128, D=256, Hs=128, Ht=128, tgt_layers=2, U_max=9, W=6)
    dw.joint.out.bias[0] += np.float32(3.0)
    e = torch.from_numpy(synth.Stream(33).normal("e", (100, 3, 256)).astype(np.float32)).cuda()
    a, b = Bd.Decoder(dw), Bd.Decoder(dw)
    want = b.decode(e)
    a.alloc_state(3, 6, 109)
    big = torch.zeros(a.prepared.numel() + 32, dtype=torch.uint8, device="cuda")
    a.prepared = big[16:16 + a.prepared.numel()]
    n = a.tables[0].numel()
    lib, m = Bd.lib(), C.byref(a.model)
    at = lambda t, o=0: C.c_void_p(t.data_ptr() + o)
    assert lib.q4_prepare_model(m, at(a.prepared), C.c_size_t(a.prepared.numel()), None) == 0 and not a.model.tables
    assert lib.q4_prepare_tables(m, at(a.tables[0], 16), C.c_size_t(n), None) != 0            # not at a 32-byte boundary
    assert lib.q4_prepare_tables(m, at(a.tables[0]), C.c_size_t(n - 1), None) != 0
    assert lib.q4_prepare_tables(m, at(a.tables[0]), C.c_size_t(n), None) == 0 and a.model.tables
    torch.cuda.synchronize()
    for x, y in zip(a.decode(e), want):
        assert torch.equal(x, y)
    for k in ("bp_parent", "bp_token", "bp_score", "pred_c", "tgt_c0"):
        assert torch.equal(a.tensors[k], b.tensors[k]), k
