"""Parity of the CUDA decoding path (through the C ABI) with the CPU oracle, step by step."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import polestar_oracle as O
from paper_2607_14107_b200 import binding as Bd
from paper_2607_14107_b200 import inputs as I
from parity import (TOL, argmax_margin_ok, check_commit_quantities, close, close_scaled, commit_margins, new_stats,
                    topk_margin_ok)

pytestmark = pytest.mark.gpu


def setup(name, std=0.02, **kw):
    m, p = I.config(name)
    model_kw = kw.pop("model", None)        # overrides of the model's shape
    if model_kw:
        m = dataclasses.replace(m, **model_kw)
    kw["flags"] = kw.get("flags", p.flags) | I.FLAG_KEEP_HIDDEN
    p = dataclasses.replace(p, **kw)
    w = I.make_weights(m, seed=0, std=std)
    wn = I.weights_to_numpy(w)
    prompt = I.make_prompt(m, p)
    gpu = Bd.Polestar(m, Bd.pack_weights(m, w), p, prompt.numpy())
    ora = O.PolestarOracle(m, wn, p, prompt.numpy())
    return m, p, gpu, ora


def check_quantised_rows(h_gpu, seq, l, tol, seen, what):
    """Rows of the NVFP4 residual cache (Appendix "Quantization Format").  The codes are integer decisions taken on
    hidden states that agree with the oracle's only within the tolerance, so a value next to a decision boundary may
    land on the neighbouring code (and a group maximum next to an E4M3 boundary on the neighbouring scale).  Hence:
    every element within the tolerance plus one code step (2 * scale, with 15% for a neighbouring scale) of the
    oracle's stored value, and all but a small share of them within the tolerance itself."""
    ref = seq.Z0[l][seq.labels[l]]
    res = (np.asarray(seq.Hc[l]) - ref).reshape(len(ref), -1, 16)
    step = np.repeat(np.abs(res).max(axis=2) / 6.0 * 2.0 * 1.15, 16, axis=1)
    err = np.abs(h_gpu - seq.Hc[l])
    base = tol + tol * np.abs(seq.Hc[l])
    assert (err <= base + step).all(), f"{what}: max abs err {err.max():.3e}"
    seen["q_elems"] = seen.get("q_elems", 0) + err.size
    seen["q_off"] = seen.get("q_off", 0) + int((err > base).sum())


def impose_codes(gpu, ora, p, m):
    """The oracle's NVFP4 codes of the rows its last step encoded, imposed on the CUDA path: a value next to a code
    boundary may fall either way when the two sides' hidden states differ in the last places."""
    d, Wm = m.d_model, gpu.W_max
    for l in range(m.n_layers):
        mask = np.zeros((p.batch, Wm), np.uint8)
        codes = np.zeros((p.batch, Wm, d // 2), np.uint8)
        scales = np.zeros((p.batch, Wm, d // 16), np.uint8)
        for s in range(p.batch):
            hc = ora.seqs[s].trace.get("hcodes", {}).get(l)
            if hc is None or len(hc[0]) == 0:
                continue
            idx, cq, sq = hc
            cq = np.asarray(cq).astype(np.uint8) & 15
            mask[s, idx] = 1
            codes[s, idx] = cq[:, 0::2] | (cq[:, 1::2] << 4)
            scales[s, idx] = torch.from_numpy(np.ascontiguousarray(sq, np.float32)).to(torch.float8_e4m3fn).view(torch.uint8).numpy()
        if mask.any():
            gpu.force_hcodes(l, mask, codes, scales)


def own_selection(gpu, m, p):
    """The CUDA path's selected window rows of the last step, per sequence and layer."""
    sel = [[] for _ in range(p.batch)]
    for l in range(m.n_layers):
        cnt, idx = gpu.read(Bd.READ_SEL_COUNT, l), gpu.read(Bd.READ_SEL_IDX, l)
        for s in range(p.batch):
            sel[s].append(idx[s, :cnt[s]].tolist())
    return sel


def run_forced(name, n_steps, std=0.02, force_labels=True, free_select=False, **kw):
    """The CUDA path replays the oracle's refresh sets and commits; every step's numbers are compared.  free_select: the CUDA
    path selects on its own (which lays the sparse forward out for the rows a selection can have) and the oracle replays that."""
    m, p, gpu, ora = setup(name, std, **kw)
    tol = TOL[m.dtype]
    L = m.n_layers
    # activations of the larger initialisations have an RMS well above one: tolerance relative to it
    close_h = close_scaled if std > 0.02 else (lambda a, b, tol, what="", depth=1: close(a, b, tol, what))
    seen = dict(refresh=0, entry_window=0, within=0, **new_stats())
    for step in range(n_steps):
        if ora.done:
            break
        if free_select and step > 0:
            info = gpu.step()
            if 0 < info.n_refreshing < p.batch:
                seen["mixed"] = seen.get("mixed", 0) + 1
            ora.step(forced_sel=own_selection(gpu, m, p))
        else:
            ora.step()     # oracle first, so that its refresh sets can be imposed on the CUDA step
        tr = ora.seqs[0].trace
        cluster = p.select_mode == I.SELECT_CLUSTER_TOPK
        if step > 0:
            if cluster and tr["kind"] != "within" and force_labels:
                # replay the oracle's clustering at later block entries (a near-tie between two centres may fall
                # either way in fp32); the first entry, inside polestar_init, is the library's own K-means
                for l in range(L):
                    lab = np.full((p.batch, gpu.W_max), 0, np.int32)
                    for s in range(p.batch):
                        lab[s, :len(ora.seqs[s].labels[l])] = ora.seqs[s].labels[l]
                    gpu.force_labels(l, lab[:, :len(ora.seqs[0].labels[l])])
            if p.flags & I.FLAG_NVFP4_HCACHE:
                impose_codes(gpu, ora, p, m)
            if not free_select:
                if tr["kind"] == "within" and tr["refresh"]:
                    for l in range(L):
                        sel = np.full((p.batch, gpu.W_max), -1, np.int32)
                        for s in range(p.batch):
                            sl = ora.seqs[s].trace["sel"][l]
                            sel[s, :len(sl)] = sl
                        gpu.force_select(l, sel)
                info = gpu.step()
            assert {0: "entry_full", 1: "entry_window", 2: "within"}[info.kind] == tr["kind"]
        if step == 0 and (p.flags & I.FLAG_NVFP4_HCACHE):
            # the first block entry ran inside polestar_init: bring its codes in line before anything reads the cache
            for s in range(p.batch):
                for l in range(L):
                    W = len(ora.seqs[s].win)
                    check_quantised_rows(gpu.read(Bd.READ_HCACHE, l)[s, :W], ora.seqs[s], l, tol, seen, f"entry H l{l}")
            impose_codes(gpu, ora, p, m)
        for s in range(p.batch):
            trs = ora.seqs[s].trace
            for l in range(L + 1):
                close_h(gpu.read(Bd.READ_HIDDEN, l)[s], trs["x_act"][l], tol, f"step {step} hidden l{l}", depth=l)
            # logits are multiplied by logit_scale, and so is their absolute error
            close_h(gpu.read(Bd.READ_LOGITS)[s] / p.logit_scale, trs["logits"] / p.logit_scale, tol, f"step {step} logits", depth=L)
            if trs["kind"] == "within":
                seen["within"] += 1
                close(gpu.read(Bd.READ_DELTA)[s], trs["delta"], tol, f"step {step} delta")
                if trs["refresh"]:
                    seen["refresh"] += 1
                    W = len(ora.seqs[s].win)
                    for l in range(L):
                        nD = len(trs["D"][l])          # window rows, or clusters (centroid proxies)
                        close(gpu.read(Bd.READ_DRIFT, l)[s, :nD], trs["D"][l], tol, f"step {step} drift l{l}")
                        n = gpu.read(Bd.READ_SEL_COUNT, l)[s]
                        assert list(gpu.read(Bd.READ_SEL_IDX, l)[s, :n]) == list(trs["sel"][l])
            elif trs["kind"] == "entry_window":
                seen["entry_window"] += 1
            if cluster and trs["kind"] != "within":
                for l in range(L):          # the clustering of this block entry
                    W = len(ora.seqs[s].win)
                    assert np.array_equal(gpu.read(Bd.READ_LABELS, l)[s, :W], ora.seqs[s].labels[l]), f"step {step} labels l{l}"
                seen["clusterings"] = seen.get("clusterings", 0) + 1
            for l in range(L):
                close_h(gpu.read(Bd.READ_KCACHE, l)[s].reshape(ora.seqs[s].Kc[l].shape), ora.seqs[s].Kc[l], tol,
                        f"step {step} K l{l}", depth=l)
                close_h(gpu.read(Bd.READ_VCACHE, l)[s].reshape(ora.seqs[s].Vc[l].shape), ora.seqs[s].Vc[l], tol,
                        f"step {step} V l{l}", depth=l)
                W = len(ora.seqs[s].win)
                if p.flags & I.FLAG_NVFP4_HCACHE:
                    # (codes imposed: only the reference rows' last-place rounding separates the stored values)
                    close(gpu.read(Bd.READ_HCACHE, l)[s, :W], ora.seqs[s].Hc[l], 1e-5, f"step {step} H l{l}")
                else:
                    close_h(gpu.read(Bd.READ_HCACHE, l)[s, :W], ora.seqs[s].Hc[l], tol, f"step {step} H l{l}", depth=l)
            _, conf = O.confidence_rows(trs["logits"], m.mask_id)
            close(gpu.read(Bd.READ_CONF)[s], conf, tol, f"step {step} conf")
        y_before = ora.tokens().copy()
        infos = ora.commit()
        forced = np.full((p.batch, p.block + gpu.W_max), -1, np.int32)
        ftok = np.zeros_like(forced)
        yh_gpu = gpu.read(Bd.READ_YHAT)
        for s, i in enumerate(infos):
            rows = np.nonzero(i["commit"] & i["masked"])[0]
            pos = [int(ora.seqs[s].act[j]) for j in rows] + i["suffix_committed"]
            forced[s, :len(pos)] = pos
            ftok[s, :len(pos)] = ora.tokens()[s, pos]
            # the CUDA path's own argmax may differ only where the oracle's two best logits nearly tie
            lg = ora.seqs[s].trace["logits"]
            for j in rows:
                if yh_gpu[s, j] != i["yhat"][j]:
                    assert abs(lg[j, yh_gpu[s, j]] - lg[j, i["yhat"][j]]) <= 2 * tol * max(1.0, p.logit_scale)
        gpu.force_commit(forced, ftok)
        ci = gpu.commit()
        assert ci.n_committed == sum(i["n_committed"] for i in infos)
        assert np.array_equal(gpu.tokens(), ora.tokens()), f"step {step} tokens"
        assert bool(ci.all_done) == ora.done
        # the commit rule itself: Delta, tau_d, the drift history and the rule's own decisions (before forcing)
        check_commit_quantities(gpu, ora, infos, y_before, p, m, tol, seen)
    gpu.destroy()
    return seen


def test_c1_forced_decisions_every_step():
    seen = run_forced("c1", 40)
    assert seen["refresh"] > 0 and seen["entry_window"] > 0
    assert seen["delta_rows"] > 0 and seen["theta_vectors"] > 20 and seen["own_by_quota"] > 0


# Workloads on which every clause of Sec. 4.2 fires in the oracle with margins above the tolerance (confidence,
# drift event, quota, suffix): larger initialisation than the default N(0, 0.02^2), whose attention rows are so
# close to uniform that their KL drift stays below the fp32 tolerance.
# The commit kernel computes in fp32 whatever the model's dtype, so its branches are pinned on the fp32 model,
# where the margins of the decisions exceed the tolerance; the bf16 model's drift values (~1e-3) lie below the bf16
# tolerance of 2e-2, so there the quantities (Delta, tau_d, history) are compared and the decisions replayed.
C1_COMMIT = dict(std=0.05, logit_scale=6.0, alpha=1.0, tau_suffix=0.5, tau_upd=2)
C1B_COMMIT = dict(logit_scale=24.0, tau_s=0.3, alpha=0.3, tau_suffix=0.3, tau_upd=-1)


def test_c1_commit_rule_branches_match_oracle():
    seen = run_forced("c1", 40, **C1_COMMIT)
    assert seen["own_by_conf"] > 0 and seen["own_by_drift"] > 0 and seen["own_by_quota"] > 0, seen
    assert seen["suffix_eligible"] > 0 and seen["own_suffix"] > 0 and seen["theta_vectors"] > 20, seen


def test_c1b_commit_quantities_match_oracle():
    seen = run_forced("c1b", 12, **C1B_COMMIT)
    assert seen["own_by_conf"] > 0 and seen["own_suffix"] > 0, seen
    assert seen["delta_rows"] > 0 and seen["theta_vectors"] > 5, seen


@pytest.mark.parametrize("name,kw", [
    ("c1", dict(tau_upd=-1, logit_scale=12.0, tau_suffix=0.5)),                      # fp32, CUDA-core attention
    ("c1b", dict(tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)),        # bf16, tensor-core attention
    ("c1b", dict(tau_upd=2, logit_scale=24.0, tau_suffix=0.5, batch=3, n_clusters=5, cluster_k=2)),
    ("c1b", dict(tau_upd=-1, logit_scale=24.0, n_clusters=16, cluster_k=16, block=8, gen_len=32, max_steps=16)),   # W = 24: ragged clusters
])
def test_centroid_proxy_mode_matches_oracle(name, kw):
    # Sec. 4.1 default policy: K-means at block entry, proxy attention of the centroids, cluster top-k -> member rows
    seen = run_forced(name, 24, select_mode=I.SELECT_CLUSTER_TOPK, **kw)
    assert seen["refresh"] >= 2 and seen["clusterings"] >= 2, seen


@pytest.mark.parametrize("name,kw,max_off", [
    ("c1", dict(tau_upd=2, logit_scale=12.0), 2e-3),
    ("c1b", dict(tau_upd=-1, logit_scale=24.0, tau_suffix=0.5, batch=3, n_clusters=5, cluster_k=2), 5e-2),
])
def test_nvfp4_hidden_cache_matches_oracle(name, kw, max_off):
    # Sec. 4.1: the window's hidden rows kept as NVFP4 residuals against the block-entry centroids; every reader
    # (proxies, recomputed rows' inputs, the next layer's packet) sees the decoded values on both sides
    m, p0 = I.config(name)
    seen = run_forced(name, 24, select_mode=I.SELECT_CLUSTER_TOPK, flags=p0.flags | I.FLAG_NVFP4_HCACHE, **kw)
    # q_off: elements of the library's own first encoding (inside polestar_init) that landed on a neighbouring code
    assert seen["refresh"] >= 2 and seen["clusterings"] >= 2 and seen["q_elems"] > 0, seen
    assert seen["q_off"] <= max_off * seen["q_elems"], seen


def test_centroid_proxy_own_clustering_matches_oracle():
    # the library's own K-means at every block entry (nothing replayed): labels equal the oracle's
    seen = run_forced("c1", 40, force_labels=False, select_mode=I.SELECT_CLUSTER_TOPK, tau_upd=2, logit_scale=12.0)
    assert seen["clusterings"] >= 2, seen


@pytest.mark.parametrize("d", [8, 40, 72, 104, 136, 168, 264, 4352])
def test_own_clustering_at_any_width(d):
    # K-means splits the columns over eight CTAs: widths that leave the last ones none (8: six of them, 40 to 168: one to three), a
    # last share that is smaller than the others (264), shares of more than 512 columns (4352).  The inputs are far from ties: the
    # oracle's largest cosine beats the next one by more than 5e-6 in every assignment (equal
    # rows apart).
    check_own_clustering("c1", 0.2, model=dict(d_model=d), batch=2)


def check_own_clustering(name, std, **kw):
    m, p, gpu, ora = setup(name, std, select_mode=I.SELECT_CLUSTER_TOPK, **kw)
    ora.step()
    for l in range(m.n_layers):
        for s in range(p.batch):
            want = ora.seqs[s].labels[l]
            assert len(want) > p.n_clusters
            assert np.array_equal(gpu.read(Bd.READ_LABELS, l)[s, :len(want)], want), (l, s)
    gpu.destroy()


@pytest.mark.parametrize("d,std", [(40, 0.02), (104, 0.01), (128, 0.01), (168, 0.01), (256, 0.01)])
def test_own_clustering_of_nearly_parallel_rows(d, std):
    # hidden rows of the second layer that differ by an angle of 1e-3 and less, as those of masked positions do: the cosines of a
    # decision differ by 5e-9 to 1e-6, and still every row goes to the centre with the largest one
    check_own_clustering("c1", std, model=dict(d_model=d), batch=2)


def test_clustering_of_rows_that_are_not_numbers():
    # a NaN embedding in the window: the row's cosines are NaN with every centre, it goes to the lowest cluster (whose
    # centre then is NaN too, so no other row stays there); behind the first attention every row is NaN
    m, p = I.config("c1")
    p = dataclasses.replace(p, select_mode=I.SELECT_CLUSTER_TOPK)
    w = I.make_weights(m, seed=0, std=0.2)
    prompt = I.make_prompt(m, p)
    bad = 37                                                   # (a window row that no centre starts from)
    tok = int(prompt.numpy().reshape(-1)[bad])
    w["embed"][tok, 5] = float("nan")
    hit = np.nonzero(prompt.numpy().reshape(-1) == tok)[0]
    gpu = Bd.Polestar(m, Bd.pack_weights(m, w), p, prompt.numpy())
    W, K = gpu.W_max, p.n_clusters
    first, second = (gpu.read(Bd.READ_LABELS, l)[0, :W] for l in range(2))
    gpu.destroy()
    starts = [(2 * j + 1) * W // (2 * K) for j in range(K)]
    assert not set(hit.tolist()) & set(starts)
    assert (first[hit] == 0).all() and (np.delete(first, hit) > 0).all() and first.max() < K
    assert (second == 0).all()


def test_c1_refresh_every_step_with_scaled_logits():
    seen = run_forced("c1", 20, tau_upd=-1, logit_scale=12.0, tau_suffix=0.5)
    assert seen["refresh"] > 10


def test_c1b_bf16_tensor_core_path():
    seen = run_forced("c1b", 16, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["refresh"] > 5


def test_c1b_bf16_norm_staging_inside_the_gemm_tail(monkeypatch):
    # opt-in variant: the RMSNorm staging of the next GEMM's input runs in the tail of the producing GEMM
    monkeypatch.setenv("POLESTAR_FUSE_PREP", "1")
    seen = run_forced("c1b", 10, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["refresh"] > 3


@pytest.mark.parametrize("variant", ["0", "5", "9", "10"])
def test_c1b_long_ragged_sequence(monkeypatch, variant):
    # N = 1100 + 64 > 1024 keys: the automatic choice (two-stream and cluster kernel), the 64-row-tile, the streaming and the
    # two-stream kernel inside the decoding loop; the prompt length is not a multiple of the block size
    monkeypatch.setenv("POLESTAR_ATTN_KERNEL", variant)
    seen = run_forced("c1b", 5, prompt_len=1100, gen_len=64, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["refresh"] >= 2


def test_c1b_bf16_rmsnorm_folded_into_the_projections(monkeypatch):
    # opt-in variant for steps without refresh: the producing projection stores x * gain and the row's sum of squares,
    # the consuming projection scales its rows (bf16 rounding before instead of after the normalisation)
    monkeypatch.setenv("POLESTAR_FOLD_NORM", "1")
    seen = run_forced("c1b", 12, tau_upd=3, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["within"] > seen["refresh"]


def test_c1b_bf16_chain_through_the_next_qkv_projection(monkeypatch):
    # opt-in: the chained kernel also stages and runs the next layer's QKV projection
    monkeypatch.setenv("POLESTAR_CHAIN_QKV", "1")
    seen = run_forced("c1b", 10, tau_upd=3, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["within"] > 0 and seen["refresh"] > 0


def test_c1b_bf16_separate_launches(monkeypatch):
    # the projections of a layer as separate launches instead of one chained kernel
    monkeypatch.setenv("POLESTAR_CHAIN", "0")
    seen = run_forced("c1b", 10, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["refresh"] > 3


GQA = dict(n_heads=8, n_kv_heads=2)


@pytest.mark.parametrize("variant,kw", [
    ("9", dict(tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=3)),
    ("9", dict(tau_upd=-1, logit_scale=24.0, tau_suffix=0.5, batch=2, select_mode=I.SELECT_CLUSTER_TOPK, n_clusters=5, cluster_k=2)),
    ("10", dict(tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=3)),
    ("10", dict(tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=2, model=GQA, prompt_len=160)),
])
def test_c1b_streaming_attention_kernel(monkeypatch, variant, kw):
    # the streaming tensor-core attention kernel (one CTA per row tile and head, two passes over the key tiles) and the two-stream
    # one on every step of a decode: block entries (recorded rows in CTAs of their own), plain steps, refresh steps with
    # stored rows / proxy rows (of the two-stream kernel: below), grouped heads
    monkeypatch.setenv("POLESTAR_ATTN_KERNEL", variant)
    seen = run_forced("c1b", 12, **kw)
    assert seen["refresh"] > 3 and seen["entry_window"] >= 0


@pytest.mark.parametrize("variant", ["9", "10"])
@pytest.mark.parametrize("prompt_len", [600, 601])          # 601: rows of 673 floats, which no bulk copy takes
def test_c1b_streaming_attention_stored_row_forms(monkeypatch, prompt_len, variant):
    # refresh steps of 24 + 72 rows over six key tiles: the first 32 rows hold the active block's and the window's stored
    # rows (row copies in the last layer, a partly recorded quarter in the others), the other quarters tensor boxes
    monkeypatch.setenv("POLESTAR_ATTN_KERNEL", variant)
    seen = run_forced("c1b", 8, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=2, prompt_len=prompt_len, gen_len=72, block=24,
                      max_steps=24)
    assert seen["refresh"] > 3


@pytest.mark.parametrize("pair_rows", [1 << 30, 1])
def test_c1b_gemm_tile_forms(monkeypatch, pair_rows):
    # the form that the default rule does not take: projections of more than 128 rows as several 128-token tiles of single
    # CTAs (devices without resident pairs), projections of up to 128 rows on CTA pairs (a pair tile's second half empty);
    # block entries of a batch (ragged: 3 x 146 and 3 x 90 rows), refresh steps (3 x 72 rows), whole and split tiles
    monkeypatch.setenv("POLESTAR_GEMM_PAIR_ROWS", str(pair_rows))
    seen = run_forced("c1b", 12, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=3, prompt_len=50, gen_len=96, block=24,
                      max_steps=16)
    assert seen["refresh"] > 3 and seen["entry_window"] > 0


@pytest.mark.parametrize("pre,suf", [(3, 1), (2, 2)])
def test_c1b_wide_windows(pre, suf):
    # refresh steps of 160 rows (32 active + 128 window rows): every projection runs on one row of pair tiles, the selection
    # rides on the O projection
    seen = run_forced("c1b", 12, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, prompt_len=128, gen_len=128, block=32,
                      max_steps=16, win_prefix_blocks=pre, win_suffix_blocks=suf)
    assert seen["refresh"] > 3 and seen["entry_window"] > 0


@pytest.mark.parametrize("variant", ["0", "10"])
@pytest.mark.parametrize("prompt_len", [616, 603])          # 603: rows of 667 floats
def test_c1b_centroid_proxies_over_more_than_512_keys(monkeypatch, prompt_len, variant):
    # the kernel that is chosen there, the two-stream one, with proxy rows as the recorded rows: block entries (684 rows a sequence, in
    # whose last layer the active block is recorded too) and refresh steps (32 + 96 + 4 rows), grouped heads
    # (initialised so that the cosines of the first entry's own clusters differ by more than bf16 moves them: 1e-4 and more)
    monkeypatch.setenv("POLESTAR_ATTN_KERNEL", variant)
    seen = run_forced("c1b", 9, std=0.05, select_mode=I.SELECT_CLUSTER_TOPK, model=GQA, batch=4, n_clusters=4, cluster_k=2, prompt_len=prompt_len,
                      tau_upd=-1, logit_scale=8.0, tau_suffix=0.5, max_steps=8)
    assert seen["refresh"] > 3 and seen["clusterings"] > 4, seen


@pytest.mark.parametrize("variant", ["0", "5"])
def test_c1b_batch_of_long_sequences_plain_steps(monkeypatch, variant):
    # 19 sequences x 8 heads, more than 1024 keys, 64-row blocks: the two-stream kernel in every step (with more (sequence, head)
    # pairs than half of the SMs plain steps have no warp-level kernel), and the 64-row warp-level kernel
    monkeypatch.setenv("POLESTAR_ATTN_KERNEL", variant)
    seen = run_forced("c1b", 7, model=dict(d_model=1024, n_heads=8, n_kv_heads=8), batch=19, prompt_len=1040, gen_len=64, block=64,
                      max_steps=16, tau_upd=5, logit_scale=12.0, alpha=0.001, tau_suffix=0.5)
    assert seen["within"] > seen["refresh"] > 0


@pytest.mark.parametrize("groups", [1, 2])
def test_c1b_epilogue_warp_groups(monkeypatch, groups):
    # projections with several token tiles drain their accumulators with four, eight or (the default) twelve warps
    monkeypatch.setenv("POLESTAR_GEMM_EPI_GROUPS", str(groups))
    seen = run_forced("c1b", 8, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=3, prompt_len=50, gen_len=96, block=24,
                      max_steps=16)
    assert seen["refresh"] > 2


def test_c1b_gemm_cta_pairs():
    # CTA pairs (tcgen05 cta_group::2: one MMA over two SMs, each loading half of the weight tile), the default for every
    # projection of more than 128 rows: ragged block entries of a batch (a pair tile's second half partly or wholly empty),
    # refresh steps, whole and split tiles, in-place L2 reductions of the O / down projections
    seen = run_forced("c1b", 12, tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, batch=3, prompt_len=50, gen_len=96, block=24,
                      max_steps=16)
    assert seen["refresh"] > 3 and seen["entry_window"] > 0


@pytest.mark.parametrize("kw", [
    dict(batch=3, prompt_len=200, gen_len=128, block=64),                                   # 768 rows of which 336: O projection on the gathered rows
    dict(batch=6, prompt_len=130, gen_len=128, block=64, tau_upd=20, tau_s=0.5),            # some sequences refresh, others do not
    dict(batch=1, prompt_len=300, gen_len=256, block=128),                                  # 384 window rows: radix selection, 512 rows of which 224
    dict(batch=1, prompt_len=128, gen_len=128, block=32, win_prefix_blocks=3),              # 160 rows: the selection rides on a pair launch
    dict(batch=3, prompt_len=200, gen_len=128, block=64, select_mode=I.SELECT_TOPK_COUNT, select_k=10 ** 6),
    dict(batch=3, prompt_len=200, gen_len=128, block=64, select_mode=I.SELECT_TOPK_COUNT, select_k=17),
    dict(batch=3, prompt_len=200, gen_len=128, block=64, select_mode=I.SELECT_TOPK_COUNT, select_k=-3),
    dict(batch=3, prompt_len=200, gen_len=128, block=64, select_mode=I.SELECT_THRESHOLD, select_thresh=1e-3),
])
def test_c1b_own_selection_matches_oracle(kw):
    # refresh steps with the library's own selection: the sparse forward is laid out for the rows that can be selected
    kw = {**dict(tau_upd=-1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5, max_steps=32), **kw}
    seen = run_forced("c1b", 5, free_select=True, **kw)
    assert seen["refresh"] >= 2, seen
    if kw["tau_upd"] >= 0:
        assert seen["mixed"] > 0, seen


def test_block_entry_of_a_large_batch_with_a_wide_feed_forward_network():
    # 64 sequences x 1024 positions x 2 * 18944 features: 37 888 pair tiles in the gate/up projection of the block entry
    m, p = I.config("c1b")
    m = dataclasses.replace(m, n_layers=1, d_ffn=18944)
    p = dataclasses.replace(p, batch=64, prompt_len=960, gen_len=64, block=32, max_steps=32)
    packed, prompt = Bd.pack_weights(m, I.make_weights(m)), I.make_prompt(m, p).numpy()
    whole = Bd.Polestar(m, packed, p, prompt)
    logits = whole.read(Bd.READ_LOGITS)
    for s in (0, 31, 63):
        one = Bd.Polestar(m, packed, dataclasses.replace(p, batch=1), prompt[s:s + 1])
        close(logits[s], one.read(Bd.READ_LOGITS)[0], TOL[m.dtype], f"sequence {s}")
        one.destroy()
    whole.commit()
    whole.step()
    whole.commit()
    whole.destroy()


def test_c1b_bf16_simt_gemm_path():
    run_forced("c1b", 6, tau_upd=-1, flags=I.FLAG_DEFAULT | Bd.FLAG_SIMT_GEMM)


@pytest.mark.parametrize("batch,prompt_len,gen_len,block", [(3, 50, 48, 16), (5, 33, 64, 32), (2, 100, 24, 8)])
def test_c1b_odd_shapes(batch, prompt_len, gen_len, block):
    # bf16 tensor-core path with batches, prompt lengths and block sizes that leave ragged row counts everywhere
    # (48 / 160 / 16 rows in the chained projections, window rows of several sequences in the sparse forward)
    seen = run_forced("c1b", 8, batch=batch, prompt_len=prompt_len, gen_len=gen_len, block=block, max_steps=gen_len // 2,
                      tau_upd=1, logit_scale=24.0, alpha=0.001, tau_suffix=0.5)
    assert seen["within"] > 0


def test_c1_batch2_gqa():
    m, p = I.config("c1")
    m = dataclasses.replace(m, n_kv_heads=2)
    p = dataclasses.replace(p, batch=2, flags=p.flags | I.FLAG_KEEP_HIDDEN, tau_upd=1)
    w = I.make_weights(m, seed=0)
    prompt = I.make_prompt(m, p)
    gpu = Bd.Polestar(m, Bd.pack_weights(m, w), p, prompt.numpy())
    ora = O.PolestarOracle(m, I.weights_to_numpy(w), p, prompt.numpy())
    ora.step()
    gpu.commit(); ora.commit()
    for step in range(10):
        gpu.step(); ora.step()
        for s in range(2):
            close(gpu.read(Bd.READ_LOGITS)[s], ora.seqs[s].trace["logits"], 1e-4, f"step {step} seq {s}")
        gpu.commit(); ora.commit()
        assert np.array_equal(gpu.tokens(), ora.tokens())


@pytest.mark.parametrize("name,kw", [("c1", C1_COMMIT), ("c1b", C1B_COMMIT)])
def test_free_running_matches_oracle(name, kw):
    """Both sides take their own decisions.  Where the oracle's decision has a margin above the tolerance the
    CUDA path must take the same one; a low-margin decision (two correct implementations may differ there) is
    replayed from the oracle for that step only, and the comparison goes on to the end of the decode."""
    m, p, gpu, ora = setup(name, **kw)
    tol = TOL[m.dtype]
    L = m.n_layers
    free = dict(select=0, commit=0)
    tot = dict(n_by_conf=0, n_by_drift=0, n_by_quota=0, n_suffix=0)
    stats = new_stats()
    first = True
    while not ora.done:
        ora.step()
        tr = ora.seqs[0].trace
        refresh = tr["kind"] == "within" and tr["refresh"]
        forced_sel = refresh and not all(topk_margin_ok(tr["D"][l], tr["sel"][l], tol) for l in range(L))
        if forced_sel:
            for l in range(L):
                sel = np.full((1, gpu.W_max), -1, np.int32)
                sel[0, :len(tr["sel"][l])] = tr["sel"][l]
                gpu.force_select(l, sel)
        if not first:
            gpu.step()
        first = False
        close_scaled(gpu.read(Bd.READ_LOGITS)[0] / p.logit_scale, tr["logits"] / p.logit_scale, tol, "logits", depth=L)
        if refresh:
            W = len(ora.seqs[0].win)
            for l in range(L):
                close(gpu.read(Bd.READ_DRIFT, l)[0, :W], tr["D"][l], tol, "drift")
                n = gpu.read(Bd.READ_SEL_COUNT, l)[0]
                assert list(gpu.read(Bd.READ_SEL_IDX, l)[0, :n]) == list(tr["sel"][l])
            free["select"] += 0 if forced_sel else 1
        y_before = ora.tokens().copy()
        info = ora.commit()[0]
        within = bool(ora.seqs[0].within)
        dec, quota_ok = commit_margins(info, p, tol, within)
        rows = np.nonzero(info["commit"] & info["masked"])[0]
        tol_logit = tol * max(1.0, p.logit_scale)
        sure = bool(dec.all()) and quota_ok and bool(argmax_margin_ok(tr["logits"], info["yhat"], m.mask_id, tol_logit)[rows].all())
        if "suffix_conf" in info:
            sc = np.asarray(info["suffix_conf"], np.float64)
            sure = sure and bool((np.abs(sc - p.tau_suffix) > tol * (1 + np.abs(sc))).all())
            sure = sure and bool(argmax_margin_ok(tr["suffix_logits"], info["suffix_yhat"], m.mask_id, tol_logit).all())
        if not sure:
            pos = [int(ora.seqs[0].act[j]) for j in rows] + info["suffix_committed"]
            forced = np.full((1, p.block + gpu.W_max), -1, np.int32)
            ftok = np.zeros_like(forced)
            forced[0, :len(pos)] = pos
            ftok[0, :len(pos)] = ora.tokens()[0, pos]
            gpu.force_commit(forced, ftok)
        ci = gpu.commit()
        assert np.array_equal(gpu.tokens(), ora.tokens())
        assert bool(ci.all_done) == ora.done
        check_commit_quantities(gpu, ora, [info], y_before, p, m, tol, stats)
        if sure:
            free["commit"] += 1
            flags = gpu.read(Bd.READ_COMMIT)[0]
            assert np.array_equal((flags & 1).astype(bool), info["commit"] & info["masked"])
            assert (ci.n_by_conf, ci.n_by_drift, ci.n_by_quota, ci.n_suffix) == \
                   (info["n_by_conf"], info["n_by_drift"], info["n_by_quota"], info["n_suffix"])
        for k in tot:      # labels come from the CUDA rule's own decision also when the positions were replayed
            tot[k] += getattr(ci, k)
    assert not (gpu.tokens() == m.mask_id).any()
    assert tot["n_by_conf"] > 0 and tot["n_by_quota"] > 0 and tot["n_suffix"] > 0, tot
    assert stats["own_by_conf"] > 0 and stats["theta_vectors"] > 0, stats
    if m.dtype == I.DTYPE_F32:
        # fp32 margins are far above the arithmetic error: most steps run without any replayed decision, and
        # drift-event commits are among the decisions both sides took alone
        assert tot["n_by_drift"] > 0 and stats["own_by_drift"] > 0, (tot, stats)
        assert free["commit"] >= 15 and free["select"] >= 2, (free, stats)
    gpu.destroy()


def test_full_refresh_equals_nocache_on_gpu():
    """select = ALL, window = everything, refresh every step must reproduce the full-recompute
    decoder of the same library (Sec. 4.1; Sec. 3.1 baseline)."""
    m, p = I.config("c1")
    w = I.make_weights(m, seed=0)
    prompt = I.make_prompt(m, p).numpy()
    packed = Bd.pack_weights(m, w)
    pa = dataclasses.replace(p, select_mode=I.SELECT_ALL, tau_upd=-1, win_prefix_blocks=8, win_suffix_blocks=8,
                             flags=(I.FLAG_DEFAULT | I.FLAG_KEEP_HIDDEN) & ~I.FLAG_SUFFIX_COMMIT, logit_scale=25.0)
    pb = dataclasses.replace(pa, flags=pa.flags | I.FLAG_NOCACHE)
    a, b = Bd.Polestar(m, packed, pa, prompt), Bd.Polestar(m, packed, pb, prompt)
    first = True
    while True:
        if not first:
            a.step(); b.step()
        first = False
        for l in range(m.n_layers + 1):
            close(a.read(Bd.READ_HIDDEN, l), b.read(Bd.READ_HIDDEN, l), 1e-4, f"hidden l{l}")
        close(a.read(Bd.READ_LOGITS), b.read(Bd.READ_LOGITS), 1e-4, "logits")
        ia, ib = a.commit(), b.commit()
        assert np.array_equal(a.tokens(), b.tokens())
        if ia.all_done:
            break
    assert ib.all_done and ia.forwards == ib.forwards


def test_zero_drift_refreshes_nothing_on_gpu():
    m, p, gpu, ora = setup("c1", tau_upd=-1)
    gpu.force_commit(np.full((1, 4), -1, np.int32))       # commit nothing at entry
    gpu.commit()
    K0 = [gpu.read(Bd.READ_KCACHE, l).copy() for l in range(m.n_layers)]
    info = gpu.step()
    assert info.kind == 2 and info.n_refreshing == 1
    for l in range(m.n_layers):
        assert gpu.read(Bd.READ_SEL_COUNT, l)[0] == 0
        assert np.abs(gpu.read(Bd.READ_DRIFT, l)).max() < 1e-5
        assert np.array_equal(gpu.read(Bd.READ_KCACHE, l), K0[l])
    assert np.abs(gpu.read(Bd.READ_DELTA)).max() < 1e-5


def test_call_order_errors():
    m, p, gpu, ora = setup("c1")
    with pytest.raises(Bd.PolestarError) as e:
        gpu.step()                                        # commit pending after init
    assert e.value.code == Bd.E_STATE
    gpu.commit()
    with pytest.raises(Bd.PolestarError) as e:
        gpu.commit()
    assert e.value.code == Bd.E_STATE
    while True:
        gpu.step()
        if gpu.commit().all_done:
            break
    with pytest.raises(Bd.PolestarError) as e:
        gpu.step()
    assert e.value.code == Bd.E_DONE
    assert not (gpu.tokens() == m.mask_id).any()


@pytest.mark.parametrize("kw", [
    dict(d_model=200, n_heads=3, n_kv_heads=1, head_dim=40, d_ffn=328, vocab=1030, mask_id=1029, eos_id=1028),     # K of 200 / 120 / 328: a last slice of 8, 56, 8; N % 32 != 0
    dict(d_model=64, n_heads=1, n_kv_heads=1, head_dim=32, d_ffn=8, vocab=34, mask_id=33, eos_id=32),          # a single slice of 64, 32 and 8; fewer columns than a tile
    dict(d_model=512, n_heads=2, n_kv_heads=2, head_dim=96, d_ffn=1096, vocab=514, mask_id=513, eos_id=512),     # more slices than the operand ring holds
])
def test_c1_projection_edges(kw):
    # fp32 projections: remainders of the K slices and of the 16 x 32 tiles (block 20: 20 and 80 rows), GQA
    seen = run_forced("c1", 8, model=kw, tau_upd=1, logit_scale=12.0, prompt_len=37, gen_len=40, block=20, max_steps=8)
    assert seen["refresh"] > 0


@pytest.mark.parametrize("frac", [0.0, 0.25, 1.0])
@pytest.mark.parametrize("batch", [1, 3, 6])          # from 3 on the O projection runs on the gathered rows
def test_c1b_free_selection_equals_the_same_selection_imposed(batch, frac):
    # an imposed selection lays the feed-forward projections out for every row of the step, a top-k selection for the rows
    # it can have: the same rows must come out (the order in which partial products meet differs, hence bf16 tolerance)
    m, p = I.config("c1b")
    p = dataclasses.replace(p, batch=batch, prompt_len=70, gen_len=128, block=64, max_steps=16, tau_upd=-1, select_frac=frac)
    packed, prompt = Bd.pack_weights(m, I.make_weights(m)), I.make_prompt(m, p).numpy()
    free, imposed = Bd.Polestar(m, packed, p, prompt), Bd.Polestar(m, packed, p, prompt)
    free.commit()
    got = free.tokens()[:, p.prompt_len:]
    pos = np.full((batch, p.gen_len), -1, np.int32)
    tok = np.full((batch, p.gen_len), -1, np.int32)
    for s in range(batch):              # near-ties of random logits may fall either way: both sides commit the same tokens
        done = np.nonzero(got[s] != m.mask_id)[0]
        pos[s, :len(done)], tok[s, :len(done)] = p.prompt_len + done, got[s, done]
    imposed.force_commit(pos, tok)
    imposed.commit()
    assert np.array_equal(free.tokens(), imposed.tokens())
    free.step()
    for l in range(m.n_layers):
        cnt, idx = free.read(Bd.READ_SEL_COUNT, l), free.read(Bd.READ_SEL_IDX, l)
        sel = np.full((batch, free.W_max), -1, np.int32)
        for s in range(batch):
            sel[s, :cnt[s]] = idx[s, :cnt[s]]
        assert cnt.max() <= int(frac * free.W_max + 0.5)
        imposed.force_select(l, sel)
    imposed.step()
    for what in (Bd.READ_LOGITS, Bd.READ_KCACHE, Bd.READ_VCACHE):
        a, b = free.read(what, m.n_layers - 1 if what != Bd.READ_LOGITS else 0), imposed.read(what, m.n_layers - 1 if what != Bd.READ_LOGITS else 0)
        close(a, b, TOL[m.dtype], f"{what}")
    free.destroy(); imposed.destroy()
