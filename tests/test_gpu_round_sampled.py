"""GPU parity of the temperature-T round (retrace_round_sampled) vs the oracle.

The verification part equals retrace_verify_sampled bit for bit (same
kernels) and the oracle's speculative sampling on every sequence whose
decisions are not within rounding of a boundary (helpers in sampling.py).
The conditioning part is a deterministic function of the accepted lengths:
it is checked against the oracle's Eq. 4-8 evaluated at the GPU's A_b.
"""

import numpy as np
import pytest
import torch

import oracle
from parity import assert_close, host_f64, host_int
from sampling import conditioned_uniforms
from paper_2608_29748_gb300.workloads import CONFIGS, make_round_inputs, make_sampled_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    from paper_2608_29748_gb300 import binding

    return binding


def conditioned_uniforms_for(x, s, seqs=None):
    sel = slice(None) if seqs is None else list(seqs)
    tl, dl = host_f64(x["logits"][sel]), host_f64(s["draft_logits"][sel])
    draft = host_int(s["draft"][sel])
    u, amb = conditioned_uniforms(tl, dl, draft, s["uniforms"][sel].cpu().numpy().astype(np.float64),
                                  s["temperature"], s["top_k"], s["top_p"])
    return tl, dl, draft, u, amb


def standalone_verify(rt, x, s, ws):
    B, K1, _ = x["logits"].shape
    outs = [torch.empty(B, dtype=torch.int32, device="cuda"), torch.empty(B, K1, dtype=torch.int32, device="cuda"),
            torch.empty(B, dtype=torch.int32, device="cuda")]
    rt.retrace_verify_sampled(x["logits"], s["draft_logits"], s["draft"], s["uniforms"], s["temperature"],
                              s["top_k"], s["top_p"], *outs, ws)
    return outs


def check_conditioning(x, out, rows, dtype):
    A = host_int(out.accept_len)
    ref = oracle.conditioned_rows(rows, A, host_f64(x["hD"]), host_f64(x["hT"]), host_f64(x["e"]),
                                  host_f64(x["Wc"]), host_f64(x["Wv"]), host_f64(x["Wg"]), x["beta"], dtype)
    got = torch.stack([out.e_out[b, j] for b, j in rows])
    assert_close(got, ref, "sampled round e~")


def check_round(rt, x, s, ws=None):
    cfg_B, K1, _ = x["logits"].shape
    K = K1 - 1
    d = x["hD"].shape[2]
    dtype = "bf16" if x["logits"].dtype == torch.bfloat16 else "f32"
    tl, dl, draft, u, amb = conditioned_uniforms_for(x, s)
    s = dict(s, uniforms=torch.tensor(u, dtype=torch.float32, device="cuda"))
    if ws is None:
        ws = rt.Workspace(cfg_B, K, x["logits"].shape[2], d, x["logits"].dtype)
    out = rt.run_round_sampled(x, s, ws)
    torch.cuda.synchronize()
    assert ws.check() == 0
    # verification: the standalone kernels' outputs, and the oracle's where unambiguous
    alone = standalone_verify(rt, x, s, ws)
    torch.cuda.synchronize()
    for a, b in zip((out.accept_len, out.committed, out.bonus), alone):
        assert torch.equal(a, b)
    want = oracle.verify_sampled(tl, dl, draft, u, s["temperature"], s["top_k"], s["top_p"])
    exact = [b for b in range(cfg_B) if b not in amb]
    np.testing.assert_array_equal(host_int(out.accept_len)[exact], want["accept_len"][exact])
    np.testing.assert_array_equal(host_int(out.committed)[exact], want["committed"][exact])
    A = host_int(out.accept_len)
    n = oracle.carried_rows(A, K)
    np.testing.assert_array_equal(host_int(out.n), n)
    # conditioning at the GPU's A_b (Eq. 4-8, batched): every row
    hD, hT = host_f64(x["hD"]), host_f64(x["hT"])
    m, uu = oracle.align(hD, hT, A)
    e_full = np.broadcast_to(host_f64(x["e"]), hD.shape)
    _, e_tilde = oracle.condition(e_full, m, uu, n, host_f64(x["Wc"]), host_f64(x["Wv"]), host_f64(x["Wg"]),
                                  x["beta"], "corrected", round_r_bf16=(dtype == "bf16"))
    assert_close(out.e_out, e_tilde, "sampled round e~")
    got = host_f64(out.e_out)
    for b in range(cfg_B):  # rows without a signal keep e bit for bit
        assert np.array_equal(got[b, n[b]:], np.broadcast_to(host_f64(x["e"]), hD.shape)[b, n[b]:])
    return out


@pytest.mark.parametrize("cfg_id", [1, 3, 4])
def test_sampled_round_matches_the_oracle(rt, cfg_id):
    cfg = CONFIGS[cfg_id]
    x = make_round_inputs(cfg, device="cuda")
    s = make_sampled_inputs(cfg, x["logits"], device="cuda")
    out = check_round(rt, x, s)
    if cfg.B > 1:
        assert 0 < host_int(out.n).sum()  # some sequences carry a rejected suffix


def test_sampled_round_dense_e_and_short_blocks(rt):
    """Per-position e (packed by the finalize kernel) and blocks of 1 and 2 drafts,
    on the tensor-core (d = 512, and 320: ragged tiles) and FFMA (d = 325)
    conditioning paths."""
    for K, d in ((1, 512), (2, 512), (16, 512), (16, 320), (16, 325)):
        cfg = CONFIGS[2].__class__("t", 9, K, 3001, d, "bf16", 1.0, "uniform", seed_offset=17)
        x = make_round_inputs(cfg, device="cuda")
        x["e"] = (torch.randn((cfg.B, K, cfg.d), device="cuda") * 0.02).to(torch.bfloat16)
        s = make_sampled_inputs(cfg, x["logits"], device="cuda")
        out = check_round(rt, x, s)
        if K == 1:
            assert torch.equal(out.e_out, x["e"])


def planted_sampling(x, accept, seed):
    """Drafts that the temperature-1 test accepts up to accept[b] whatever the
    uniforms (the target's most likely tokens, then one outside the vocabulary)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, K1, V = x["logits"].shape
    K = K1 - 1
    draft = torch.argmax(x["logits"][:, :K].float(), dim=-1).to(torch.int32)
    for b, a in enumerate(accept):
        if a < K:
            draft[b, a] = V
    noise = torch.randn((B, K, V), generator=g, device="cuda")
    uniforms = torch.rand((B, K1), generator=g, device="cuda") * 0.01
    uniforms[:, K] = torch.rand((B,), generator=g, device="cuda")
    return {"draft_logits": (x["logits"][:, :K].float() + 0.1 * noise).to(x["logits"].dtype), "draft": draft,
            "uniforms": uniforms, "temperature": 1.0, "top_k": 20, "top_p": 0.95}


@pytest.mark.parametrize("windows", [False, True])
@pytest.mark.parametrize("B,K,V,d", [(1, 16, 4099, 2560), (4, 16, 1003, 264), (8, 8, 515, 512), (2, 33, 300, 136), (1, 65, 64, 256),
                                     (2, 8, 333, 4352)])
def test_sampled_rounds_of_few_sequences(rt, B, K, V, d, windows):
    """At most 64 tile rows and a broadcast e: the conditioning reads the carried
    rows where they lie, by the accepted lengths that the finalize kernel wrote.
    A = 0, K - 2, K - 1 and K, on one workspace with greedy rounds between (which
    decide the sequences from the argmax keys there)."""
    cfg = CONFIGS[2].__class__("few", B, K, V, d, "bf16", 1.0, "uniform", seed_offset=B + K)
    x = make_round_inputs(cfg, device="cuda")
    ws = rt.Workspace(B, K, V, d, torch.bfloat16)
    prev = rt.retrace_set_verify_schedule(rt.VERIFY_WINDOWS if windows else rt.VERIFY_FULL)
    try:
        greedy = rt.run_round(x, rt.Workspace(B, K, V, d, torch.bfloat16))
        for shift in range(4):
            accept = [[0, K - 2, K - 1, K][(b + shift) % 4] for b in range(B)]
            out = check_round(rt, x, planted_sampling(x, accept, shift), ws)
            assert host_int(out.accept_len).tolist() == accept
            between = rt.run_round(x, ws)
            torch.cuda.synchronize()
            assert torch.equal(between.committed, greedy.committed) and torch.equal(between.e_out, greedy.e_out)
    finally:
        rt.retrace_set_verify_schedule(prev)
    assert ws.check() == 0


@pytest.mark.parametrize("dense_e", [False, True])
@pytest.mark.parametrize("d", [256, 264])
def test_sampled_rounds_of_many_rows(rt, d, dense_e):
    """Above the small-R line: the rows that the finalize kernel packed, in the
    CTA-pair kernel (whole and ragged tiles, per-position e) and the one-SM kernel
    (per-position e, d a multiple of 256)."""
    cfg = CONFIGS[2].__class__("many", 274, 16, 515, d, "bf16", 1.0, "uniform", seed_offset=d)
    x = make_round_inputs(cfg, device="cuda")
    if dense_e:
        x["e"] = (torch.randn((cfg.B, cfg.K, cfg.d), device="cuda") * 0.02).to(torch.bfloat16)
    accept = [(5 * b) % (cfg.K + 1) for b in range(cfg.B)]
    out = check_round(rt, x, planted_sampling(x, accept, d))
    assert host_int(out.accept_len).tolist() == accept


def test_sampled_round_serving_batch(rt):
    """Config 5 at full size (B=256, K=16, V=151936, d=4096) in the launch
    configuration the benchmark times: verification on a seeded sample of
    sequences against the oracle, every unconditioned row, and a sample of
    conditioned rows."""
    cfg = CONFIGS[5]
    x = make_round_inputs(cfg, device="cuda")
    s = make_sampled_inputs(cfg, x["logits"], device="cuda")
    ws = rt.Workspace(cfg.B, cfg.K, cfg.V, cfg.d, cfg.torch_dtype)
    out = rt.run_round_sampled(x, s, ws)
    alone = standalone_verify(rt, x, s, ws)
    torch.cuda.synchronize()
    assert ws.check() == 0
    for a, b in zip((out.accept_len, out.committed, out.bonus), alone):
        assert torch.equal(a, b)
    rng = np.random.default_rng(11)
    seqs = sorted(rng.choice(cfg.B, size=8, replace=False).tolist())
    tl, dl, draft, u, amb = conditioned_uniforms_for(x, s, seqs)
    s2 = {k: (v[seqs].contiguous() if torch.is_tensor(v) else v) for k, v in s.items()}
    s2["uniforms"] = torch.tensor(u, dtype=torch.float32, device="cuda")
    x2 = {k: (v[seqs].contiguous() if torch.is_tensor(v) and v.dim() == 3 else v) for k, v in x.items()}
    sub = rt.run_round_sampled(x2, s2, rt.Workspace(len(seqs), cfg.K, cfg.V, cfg.d, cfg.torch_dtype))
    torch.cuda.synchronize()
    want = oracle.verify_sampled(tl, dl, draft, u, s["temperature"], s["top_k"], s["top_p"])
    exact = [i for i in range(len(seqs)) if i not in amb]
    np.testing.assert_array_equal(host_int(sub.accept_len)[exact], want["accept_len"][exact])
    np.testing.assert_array_equal(host_int(sub.committed)[exact], want["committed"][exact])
    n = oracle.carried_rows(host_int(out.accept_len), cfg.K)
    np.testing.assert_array_equal(host_int(out.n), n)
    assert 0 < n.sum()
    pos = torch.arange(cfg.K, device="cuda")[None, :]
    mask = pos >= out.n.long()[:, None]
    assert torch.equal(out.e_out[mask], x["e"].expand(int(mask.sum()), cfg.d))
    cond = [(b, j) for b in range(cfg.B) for j in range(int(n[b]))]
    pick = sorted({0, len(cond) - 1, *rng.choice(len(cond), size=40, replace=False).tolist()})
    check_conditioning(x, out, [cond[i] for i in pick], "bf16")


def test_sampled_round_in_cuda_graph(rt):
    """The sampled round captures into a CUDA graph and replays exactly."""
    cfg = CONFIGS[4]
    x = make_round_inputs(cfg, device="cuda")
    s = make_sampled_inputs(cfg, x["logits"], device="cuda")
    ws = rt.Workspace(cfg.B, cfg.K, cfg.V, cfg.d, cfg.torch_dtype)
    eager = rt.run_round_sampled(x, s, ws)
    torch.cuda.synchronize()
    out = rt.RoundBuffers(cfg.B, cfg.K, cfg.d, cfg.torch_dtype)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        rt.run_round_sampled(x, s, ws, out=out, stream=st)
    torch.cuda.current_stream().wait_stream(st)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        rt.run_round_sampled(x, s, ws, out=out, stream=st)
    for _ in range(2):
        out.e_out.zero_()
        g.replay()
    torch.cuda.synchronize()
    assert ws.check() == 0
    for a, b in ((out.accept_len, eager.accept_len), (out.committed, eager.committed), (out.n, eager.n),
                 (out.e_out, eager.e_out)):
        assert torch.equal(a, b)
