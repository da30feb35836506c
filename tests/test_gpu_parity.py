"""GPU parity: the CUDA path, called through the C ABI, against the fp64
oracle on the same seeded inputs (tolerances in tests/gpu_harness.py)."""
import json

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - GPU tests only run on the GPU machine
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2607_10582_gb300 as md  # noqa: E402
import synth  # noqa: E402
from paper_2607_10582_gb300 import build as mdbuild  # noqa: E402
from tests.attention_shapes import CLUSTER  # noqa: E402
from tests.gpu_harness import TOL_O_ABS, Lockstep, to_dev  # noqa: E402

mdbuild.build()
synth.build()


def test_cuda_generator_matches_host():
    regions = (np.arange(300) % 7).astype(np.uint8)
    for structured in (False, True):
        k, v = synth.kv_host(5, 3, 2, 2, 40, 300, regions, structured)
        kd = torch.empty(k.shape, dtype=torch.int16, device="cuda")
        vd = torch.empty(v.shape, dtype=torch.int16, device="cuda")
        rd = torch.from_numpy(regions).cuda()
        kap = (synth.ctypes.c_float * 9)(*synth.KAPPA_STRUCT) if structured else None
        assert synth.lib().synth_fill_kv_dev(5, int(structured), kap, 3, 2, 2, 128, 40, 300,
                                             rd.data_ptr(), kd.data_ptr(), vd.data_ptr(), None) == 0
        torch.cuda.synchronize()
        assert np.array_equal(kd.cpu().numpy().view(np.uint16), k)
        assert np.array_equal(vd.cpu().numpy().view(np.uint16), v)
    q = synth.q_host(9, 3, 2, 12, 2, 11, True)
    qd = torch.empty(q.shape, dtype=torch.int16, device="cuda")
    kap = (synth.ctypes.c_float * 9)(*synth.KAPPA_STRUCT)
    assert synth.lib().synth_fill_q_dev(9, 1, kap, 3, 2, 12, 6, 128, 11, qd.data_ptr(), None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(qd.cpu().numpy().view(np.uint16), q)


def report(name, ls):
    """One line per lockstep run: largest errors, the choices adopted inside
    the tie band and how close the decisions came to the band (TieStats)."""
    print("\nLOCKSTEP " + json.dumps({"run": name, "max_err": ls.max_err, "resyncs": ls.resyncs,
                                      "ties": ls.ties.summary()}))


def test_config0_full_run():
    """Config 0 end to end: 448-token trace, 64 decode steps, eviction to 50%
    of pages at every step."""
    ls = Lockstep(synth.make_workload(0)).run()
    ls.check_layout()
    assert ls.max_err["O"] < 2e-2
    report("config 0", ls)


def test_multichunk_ragged_batch():
    """Ragged sequences long enough to split each (layer, head) item into many
    chunks, GQA group 8, pages of 16 with partial last pages."""
    w = synth.custom_workload("ragged", L=2, Hq=16, Hkv=2, page_size=16,
                              lengths=[37, 1300, 5003], budget_frac=0.4, steps=12, seed=3)
    ls = Lockstep(w).run()
    ls.check_layout()


def test_group6_page32_structured():
    """Group of 6 query heads (padded to 8 in the kernel), pages of 32, keys
    and queries with region structure and hot tokens so refreshes fire."""
    w = synth.custom_workload("g6", L=3, Hq=12, Hkv=2, page_size=32, lengths=[700, 2100],
                              budget_frac=0.5, steps=12, seed=4, structured=True)
    ls = Lockstep(w).run()
    ls.check_layout()


@pytest.mark.parametrize("Hq,Hkv,ps", [(4, 4, 16), (4, 2, 32), (2, 1, 16)])
def test_small_gqa_groups(Hq, Hkv, ps):
    """Groups of 1 and 2 query heads per KV head (multi-head attention at
    G = 1): the kernel pads every group to 8 heads and masks the padding."""
    w = synth.custom_workload(f"g{Hq // Hkv}", L=2, Hq=Hq, Hkv=Hkv, page_size=ps, lengths=[900, 2600],
                              budget_frac=0.5, steps=6, seed=31 + Hq + Hkv, structured=True)
    ls = Lockstep(w).run()
    ls.check_layout()


def test_observation_window():
    """Observation every 4 decode steps: the mass of the window's steps is
    accumulated and averaged (Sec. III-C)."""
    w = synth.custom_workload("win", L=2, Hq=8, Hkv=2, page_size=16, lengths=[900, 600],
                              budget_frac=0.5, steps=16, seed=5, window_k=4, structured=True)
    ls = Lockstep(w).run()
    ls.check_layout()


@pytest.mark.parametrize("score_mode,page_reduce,w", [(1, 0, 4.0), (0, 1, 0.5), (1, 1, 0.0)])
def test_score_variants(score_mode, page_reduce, w):
    wl = synth.custom_workload("var", L=2, Hq=16, Hkv=2, page_size=16, lengths=[800, 1000],
                               budget_frac=0.3, steps=8, seed=6, score_mode=score_mode,
                               page_reduce=page_reduce, attn_weight=w, structured=True)
    Lockstep(wl).run().check_layout()


@pytest.mark.parametrize("mode", [2, 3, 4])
def test_policy_variants(mode):
    """Score modes beyond Eq. 4: the attention term normalised to the uniform
    level (2), recency / streaming (3), seeded random (4), and the H2O-style
    accumulated-attention configuration (mode 0, rho = gamma = 1, b = 0)."""
    w = synth.custom_workload("pol", L=2, Hq=16, Hkv=2, page_size=16, lengths=[900, 1500],
                              budget_frac=0.3, steps=8, seed=16, score_mode=mode, structured=True)
    for b in range(w.B):
        w.insert_steps[b][:] = -(np.arange(w.n0(b))[::-1] // 16)
    w.extra["random_seed"] = 99
    Lockstep(w).run().check_layout()
    if mode == 2:
        h2o = synth.custom_workload("h2o", L=2, Hq=16, Hkv=2, page_size=16, lengths=[1100],
                                    budget_frac=0.3, steps=8, seed=17, rho=1.0, gamma=1.0,
                                    base=(0.0,) * 7, pinned=(0,) * 7, structured=True)
        Lockstep(h2o).run().check_layout()


def test_region_aligned_pages():
    """Region-aligned allocation (a fresh page at each region boundary): no
    page straddles two regions, pages are partly filled, every stage masks by
    page fill, and eviction removes exactly the evicted pages' tokens."""
    w = synth.custom_workload("aligned", L=2, Hq=16, Hkv=2, page_size=16, lengths=[700, 1900],
                              budget_frac=0.5, steps=20, seed=18, structured=True)
    w.extra["region_aligned"] = True
    ls = Lockstep(w)
    ls.prefill()
    ls.check_layout()
    assert any(f < 16 for f in ls.orc.fill[0][:-1])          # partial interior pages
    for s in range(w.steps):
        ls.decode(regions=[[6, 2][s % 2]] * w.B)            # alternating regions: page per switch
        ls.observe()
    ls.check_layout()
    w2 = synth.custom_workload("aligned32", L=1, Hq=12, Hkv=2, page_size=32, lengths=[1500],
                               budget_frac=0.4, steps=8, seed=19, window_k=2)
    w2.extra["region_aligned"] = True
    Lockstep(w2, layerwise=True).run().check_layout()


def test_pins_over_budget_warns():
    """Pinned pages alone exceed the budget: every evictable page goes, the
    warning comes back, pinned pages stay."""
    w = synth.custom_workload("pins", L=1, Hq=8, Hkv=2, page_size=16, lengths=[400],
                              budget_frac=0.1, steps=2, seed=7)
    w.regions[0][:] = synth.SYSTEM
    w.regions[0][100:180] = synth.TOOL_OUT
    ls = Lockstep(w)
    ls.prefill()
    ls.decode()
    n = ls.observe()
    assert n[0] > 0
    st, _ = ls.gpu.evict([1])
    assert st == md.MD_WARN_OVER_BUDGET


def test_layer_by_layer_decode():
    """md_decode_layer, one layer per call (the shape a real model with MLPs
    between layers uses), matches the oracle's whole decode step."""
    w = synth.custom_workload("layers", L=3, Hq=16, Hkv=2, page_size=16, lengths=[500, 2200],
                              budget_frac=0.4, steps=10, seed=12, structured=True)
    ls = Lockstep(w, layerwise=True).run()
    ls.check_layout()
    w4 = synth.custom_workload("layers4", L=4, Hq=12, Hkv=2, page_size=32, lengths=[1300],
                               budget_frac=0.5, steps=6, seed=13, window_k=3)
    Lockstep(w4, layerwise=True).run().check_layout()


def test_layer_by_layer_call_order_is_enforced():
    c = md.Cache(2, 8, 2, 16, 1, 8, 16)
    z = torch.zeros((1, 8, 128), dtype=torch.int16, device="cuda")
    zk = torch.zeros((1, 2, 128), dtype=torch.int16, device="cuda")
    with pytest.raises(md.MemDecayError) as e:
        c.decode_layer(1, 1, z, zk, zk, [6], z)
    assert e.value.status == md.MD_ERR_STATE
    c.decode_layer(0, 1, z, zk, zk, [6], z)
    for call in (lambda: c.evict([4]), lambda: c.decode_layer(0, 1, z, zk, zk, [6], z)):
        with pytest.raises(md.MemDecayError) as e:
            call()
        assert e.value.status == md.MD_ERR_STATE
    c.decode_layer(1, 1, z, zk, zk, [6], z)
    st, n = c.evict([4])
    assert st == md.MD_OK and c.query(md.MD_QUERY_TOKENS, 0) == 1
    assert c.sync() == md.MD_OK


def test_calibration_histogram_and_fit():
    """The calibration by-product (Sec. IV-B, Eqs. 6-7): the region x age
    histogram of the observed mass, gathered on the GPU during observation
    steps, matches the oracle's, and so do the fitted rates."""
    w = synth.custom_workload("calib", L=2, Hq=16, Hkv=2, page_size=16, lengths=[1200, 700],
                              budget_frac=0.6, steps=24, seed=14, structured=True)
    w.insert_steps[0][:] = -np.arange(1200)[::-1] // 3      # a spread of ages
    ls = Lockstep(w, calib=True).run()
    assert ls.check_calibration() > 1000
    w3 = synth.custom_workload("calib_win", L=2, Hq=8, Hkv=2, page_size=32, lengths=[900],
                               budget_frac=0.5, steps=12, seed=15, window_k=4)
    Lockstep(w3, calib=True).run().check_calibration()


def test_config1_full_run():
    """Config 1 end to end (Qwen2.5-1.5B geometry, 28 layers, 12/2 heads):
    1,700-token trace, all 256 decode steps, eviction to 25% of the pages."""
    ls = Lockstep(synth.make_workload(1))
    ls.run()
    ls.check_layout()
    report("config 1", ls)


@pytest.mark.parametrize("structured", [False, True])
def test_config2_all_steps(structured):
    """Config 2 end to end (Qwen2.5-3B geometry, 36 layers, 16/2 heads), 32
    sequences with Dirichlet region spans and insertion offsets: the
    full-trace step and all 255 steady steps, every sequence at every step
    (page boundaries pass, so appends take pages the evictions freed).  With
    structured keys and queries (per-region offsets, hot tokens) refreshes
    fire."""
    ls = Lockstep(synth.make_workload(2, structured=structured))
    ls.run()
    ls.check_layout()
    report(f"config 2{' structured' if structured else ''}", ls)
    if structured:
        o = ls.orc
        sl = np.concatenate([o.slots(b) for b in range(ls.w.B)])
        assert np.count_nonzero((o.t_ref[sl] == o.t) & (o.t_ins[sl] < o.t)) > 0   # refreshed, not new


def _small_run(seed):
    w = synth.custom_workload("det", L=2, Hq=16, Hkv=2, page_size=16, lengths=[700, 1500],
                              budget_frac=0.5, steps=6, seed=seed, structured=True)
    c = md.Cache(w.L, w.Hq, w.Hkv, w.page_size, w.B, w.max_pages_per_seq(), w.num_phys_pages())
    for r in range(7):
        c.set_region_params(r, w.base[r], w.half_life[r], bool(w.pinned[r]))
    for b in range(w.B):
        k, v = synth.kv_host(w.seed, b, w.L, w.Hkv, 0, w.n0(b), w.regions[b], True)
        c.append_tokens(b, w.regions[b], to_dev(k), to_dev(v))
    outs = []
    pos = [w.n0(b) for b in range(w.B)]
    for t in range(1, 7):
        q = synth.q_host(w.seed, w.B, w.L, w.Hq, w.Hkv, t, True)
        kn, vn = synth.step_kv_host(w.seed, pos, [6] * w.B, w.L, w.Hkv, True)
        out = torch.empty((w.B, w.L, w.Hq, 128), dtype=torch.int16, device="cuda")
        c.decode_step(w.B, to_dev(q), to_dev(kn), to_dev(vn), [6] * w.B, out)
        c.evict(w.budget_pages)
        pos = [p + 1 for p in pos]
        outs.append(out.clone())
    states = [c.get_state(s) for s in (md.MD_STATE_A, md.MD_STATE_AHAT, md.MD_STATE_PAGE_SCORE,
                                       md.MD_STATE_BLOCK_TABLE, md.MD_STATE_FREE)]
    torch.cuda.synchronize()
    return outs, states


def test_bit_identical_reruns():
    """No float atomics anywhere: two runs give bit-identical outputs and
    state (a proxy for the absence of races)."""
    o1, s1 = _small_run(8)
    o2, s2 = _small_run(8)
    for x, y in zip(o1 + s1, o2 + s2):
        assert torch.equal(x, y)


def test_config2_full_trace_step_is_bit_identical_over_reruns():
    """The full-trace step of the 3B geometry (32 x 1,700 tokens, one split per
    (sequence, layer, KV head), several units per CTA) repeated from one saved
    state gives bit-identical outputs and step mass.  A ring stage refilled by
    TMA (async proxy) before the consumers' ldmatrix reads of it (generic
    proxy) were fenced showed up here as rare, small differences in one
    item's output (its V rows read after the refill had begun)."""
    w = synth.make_workload(2)
    dev = torch.device("cuda")
    B, L, Hq, Hkv, D = w.B, w.L, w.Hq, w.Hkv, w.D
    c = md.Cache(L, Hq, Hkv, w.page_size, B, w.max_pages_per_seq(), w.num_phys_pages())
    for r in range(7):
        c.set_region_params(r, w.base[r], w.half_life[r], bool(w.pinned[r]))
    lib = synth.lib()
    nmax = max(w.n0(b) for b in range(B))
    kb = torch.empty(L * Hkv * nmax * D, dtype=torch.int16, device=dev)
    vb = torch.empty_like(kb)
    for b in range(B):
        rd = torch.from_numpy(w.regions[b]).to(dev)
        assert lib.synth_fill_kv_dev(w.seed, 0, None, b, L, Hkv, D, 0, w.n0(b), rd.data_ptr(),
                                     kb.data_ptr(), vb.data_ptr(), None) == 0
        c.append_tokens(b, w.regions[b], kb.data_ptr(), vb.data_ptr(), w.insert_steps[b])
    q = torch.empty((B, L, Hq, D), dtype=torch.int16, device=dev)
    kn = torch.empty((B, L, Hkv, D), dtype=torch.int16, device=dev)
    vn = torch.empty_like(kn)
    pos = torch.tensor([w.n0(b) for b in range(B)], dtype=torch.int32, device=dev)
    rg = torch.tensor([w.decode_region] * B, dtype=torch.uint8, device=dev)
    assert lib.synth_fill_q_dev(w.seed, 0, None, B, L, Hq, Hq // Hkv, D, 1, q.data_ptr(), None) == 0
    assert lib.synth_fill_step_kv_dev(w.seed, 0, None, B, L, Hkv, D, pos.data_ptr(), rg.data_ptr(),
                                      kn.data_ptr(), vn.data_ptr(), None) == 0
    torch.cuda.synchronize()
    saved = c.save_state()
    ref = None
    for rep in range(16):
        c.load_state(saved)
        out = torch.empty((B, L, Hq, D), dtype=torch.int16, device=dev)
        c.decode_step(B, q, kn, vn, [w.decode_region] * B, out)
        got = (out.clone(), c.get_state(md.MD_STATE_MASS).clone())
        torch.cuda.synchronize()
        if ref is None:
            ref = got
            continue
        assert torch.equal(got[0], ref[0]), f"attention output differs on rerun {rep}"
        assert torch.equal(got[1], ref[1]), f"step mass differs on rerun {rep}"
    assert c.sync() == md.MD_OK
    c.close()


def test_decode_step_host_matches_device_path():
    """md_decode_step_host (host buffers) gives the same bits as
    md_decode_step from the same state: with pinned torch tensors and with
    pageable numpy arrays, the K/V and output buffers used in place where the
    device reaches them (the kernels read and write host memory) and through
    copies when that is switched off or a buffer is misaligned; an
    out-of-range batch is rejected before anything is copied."""
    w = synth.custom_workload("host", L=2, Hq=16, Hkv=2, page_size=16, lengths=[700, 1500],
                              budget_frac=0.5, steps=4, seed=5, structured=True)
    B, L, Hq, Hkv = w.B, w.L, w.Hq, w.Hkv
    c = md.Cache(L, Hq, Hkv, w.page_size, B, w.max_pages_per_seq(), w.num_phys_pages())
    for r in range(7):
        c.set_region_params(r, w.base[r], w.half_life[r], bool(w.pinned[r]))
    for b in range(B):
        k, v = synth.kv_host(w.seed, b, L, Hkv, 0, w.n0(b), w.regions[b], True)
        c.append_tokens(b, w.regions[b], to_dev(k), to_dev(v))
    q = np.ascontiguousarray(synth.q_host(w.seed, B, L, Hq, Hkv, 1, True))
    kn, vn = (np.ascontiguousarray(x) for x in
              synth.step_kv_host(w.seed, [w.n0(b) for b in range(B)], [6] * B, L, Hkv, True))
    regs = [6] * B
    torch.cuda.synchronize()
    saved = c.save_state()
    out_dev = torch.empty((B, L, Hq, 128), dtype=torch.int16, device="cuda")
    c.decode_step(B, to_dev(q), to_dev(kn), to_dev(vn), regs, out_dev)
    ref_o = out_dev.cpu()
    ref_m = c.get_state(md.MD_STATE_MASS).cpu()

    c.load_state(saved)
    qh, kh, vh = (torch.from_numpy(x.view(np.int16)).pin_memory() for x in (q, kn, vn))
    outh = torch.zeros((B, L, Hq, 128), dtype=torch.int16).pin_memory()
    c.decode_step_host(B, qh, kh, vh, regs, outh)
    assert c.sync() == md.MD_OK
    assert torch.equal(outh, ref_o)
    assert torch.equal(c.get_state(md.MD_STATE_MASS).cpu(), ref_m)

    c.load_state(saved)
    outn = np.zeros((B, L, Hq, 128), np.uint16)
    c.decode_step_host(B, q, kn, vn, regs, outn)
    assert c.sync() == md.MD_OK
    assert np.array_equal(outn, ref_o.numpy().view(np.uint16))

    # the copy path, pinned and pageable
    c.debug_set(md.MD_DEBUG_ZERO_COPY, 0)
    for bufs in ((qh, kh, vh), (q, kn, vn)):
        c.load_state(saved)
        outc = torch.zeros((B, L, Hq, 128), dtype=torch.int16).pin_memory()
        c.decode_step_host(B, *bufs, regs, outc)
        assert c.sync() == md.MD_OK
        assert torch.equal(outc, ref_o)
        assert torch.equal(c.get_state(md.MD_STATE_MASS).cpu(), ref_m)
    c.debug_set(md.MD_DEBUG_ZERO_COPY, 1)
    # a misaligned K buffer (2 bytes off) goes through a copy, V and the output in place
    c.load_state(saved)
    km = np.zeros(kn.size + 1, np.uint16)[1:].reshape(kn.shape)
    km[...] = kn
    assert km.ctypes.data % 16 != 0
    outm = np.zeros((B, L, Hq, 128), np.uint16)
    c.decode_step_host(B, q, km, vn, regs, outm)
    assert c.sync() == md.MD_OK
    assert np.array_equal(outm, ref_o.numpy().view(np.uint16))

    with pytest.raises(md.MemDecayError) as ei:
        c.decode_step_host(B + 1, q, kn, vn, regs + [6], outn)
    assert ei.value.status == md.MD_ERR_INVALID_ARG
    c.close()


def test_host_buffer_steps_follow_the_oracle():
    """Many decode + evict steps through md_decode_step_host with pinned
    buffers (query rows copied in, new K/V read and output written in place
    over the host link), evictions and page turnover included, against the
    oracle at every step."""
    w = synth.custom_workload("hostpath", L=2, Hq=16, Hkv=2, page_size=16, lengths=[700, 1500, 37],
                              budget_frac=0.4, steps=40, seed=23, structured=True)
    ls = Lockstep(w, host_buffers=True).run()
    ls.check_layout()


def test_entry_points_mixed_step_by_step():
    """Every kernel is launched with programmatic dependent launch, so a
    kernel may start before the one ahead of it ends and relies on waiting
    for it.  Steps that switch entry point every time (device buffers, host
    buffers, layer by layer, with an observation after each) still follow the
    oracle at every step."""
    w = synth.custom_workload("mixed", L=3, Hq=16, Hkv=2, page_size=16, lengths=[900, 40, 2100],
                              budget_frac=0.4, steps=24, seed=29, structured=True)
    ls = Lockstep(w)
    ls.prefill()
    for s in range(w.steps):
        ls.decode(entry=("device", "host", "layers")[s % 3])
        ls.observe()
        if s % 5 == 4:
            ls.check_layout()
    ls.check_layout()


@pytest.mark.parametrize("L,Hq,Hkv,ps,lengths,aligned", [shape for shape, _ in CLUSTER])
def test_cluster_attention_follows_the_oracle(L, Hq, Hkv, ps, lengths, aligned):
    """Launch shapes that take the cluster attention kernel by themselves, with
    sizes at the edges of tiles, warps and chunks."""
    w = synth.custom_workload("cluster", L=L, Hq=Hq, Hkv=Hkv, page_size=ps, lengths=lengths, budget_frac=0.7,
                              steps=3, seed=41, structured=True)
    w.extra["region_aligned"] = bool(aligned)
    ls = Lockstep(w).run()
    ls.check_layout()


@pytest.mark.parametrize("C,warps,spill,n", [
    (1, 4, 0, 1500), (2, 4, 0, 1500), (8, 4, 0, 1500), (16, 4, 0, 3000),
    (1, 8, 0, 2200), (4, 8, 0, 2200), (16, 8, 0, 5000),
    # scores in scratch: 47 and 35 tiles per warp of 4, 34 of 8 (page ids come 32
    # at a time; the new token is on the last tile), few tiles, and none
    (1, 4, 1, 3000), (2, 4, 1, 4400), (1, 8, 1, 4340), (8, 4, 1, 900), (16, 8, 1, 5000),
])
@pytest.mark.parametrize("ps,aligned", [(16, 0), (32, 0), (16, 1), (32, 1)])
def test_every_cluster_form_follows_the_oracle(C, warps, spill, n, ps, aligned):
    """Every form of the cluster kernel on the same kinds of batch (a step at
    once and layer by layer): one whose sequences fill most chunks, one that
    leaves most of them empty."""
    w = synth.custom_workload("form", L=2, Hq=12, Hkv=2, page_size=ps, lengths=[n, 17, n // 3, 1], budget_frac=0.9,
                              steps=2, seed=43, structured=True)
    w.extra["region_aligned"] = bool(aligned)
    ls = Lockstep(w)
    ls.gpu.debug_set(md.MD_DEBUG_CLUSTER_FORM, C + 256 * warps + 65536 * spill)
    ls.prefill()
    for entry in ("device", "layers"):
        ls.decode(entry=entry)
        ls.observe()
    ls.check_layout()


def test_cluster_form_that_does_not_fit_fails():
    """A forced form whose scores fit neither shared memory nor, spilled, the
    scratch is an error of the step, not another form."""
    w = synth.custom_workload("nofit", L=1, Hq=4, Hkv=1, page_size=16, lengths=[3000], budget_frac=1.0, steps=1, seed=44)
    ls = Lockstep(w)
    ls.prefill()
    ls.gpu.debug_set(md.MD_DEBUG_CLUSTER_FORM, 1 + 256 * 4)
    with pytest.raises(md.MemDecayError) as e:
        ls.decode()
    assert e.value.status == md.MD_ERR_CUDA


@pytest.mark.parametrize("Hq,Hkv,ps,lengths,aligned,window", [
    (16, 2, 16, [37, 1300, 5003], 0, 1),
    (12, 2, 32, [700, 2100], 0, 3),
    (2, 2, 16, [900, 2600], 0, 1),
    (16, 2, 16, [700, 1900, 0], 1, 1),
    (12, 2, 32, [1500, 33], 1, 2),
])
@pytest.mark.parametrize("entry", ["device", "host", "layers", "mixed"])
def test_persistent_attention_follows_the_oracle(Hq, Hkv, ps, lengths, aligned, window, entry):
    """The persistent kernel (kept by the grid limit, here all that fit) on
    shapes that take the cluster kernel by themselves: both page sizes,
    contiguous and region-aligned pages, appending inside the launch and behind
    an append launch."""
    w = synth.custom_workload("persistent", L=3, Hq=Hq, Hkv=Hkv, page_size=ps, lengths=lengths, budget_frac=0.5,
                              steps=12, seed=45, window_k=window, structured=True)
    w.extra["region_aligned"] = bool(aligned)
    ls = Lockstep(w)
    ls.gpu.debug_set(md.MD_DEBUG_GRID_LIMIT, 512)
    ls.prefill()
    for s in range(w.steps):
        ls.decode(entry=("device", "host", "layers")[s % 3] if entry == "mixed" else entry,
                  regions=[[6, 2][s // 2 % 2]] * w.B)
        if (s + 1) % window == 0:
            ls.observe()
    ls.check_layout()


@pytest.mark.parametrize("ps,aligned,window", [(16, 0, 1), (32, 0, 3), (32, 1, 1), (16, 1, 2)])
@pytest.mark.parametrize("kernel", ["by cost", "8 warps", "scratch", "persistent"])
def test_calls_back_to_back_give_what_calls_one_by_one_give(ps, aligned, window, kernel):
    """Layer calls, whole steps and evictions issued with nothing between them,
    on tensors prepared beforehand: launches overlap (layers after the first copy
    K/V before the layer ahead has ended).  Outputs, the step's mass and the
    state are the same bits as with a synchronisation after every call."""
    L, Hq, Hkv, steps = 4, 16, 2, 12
    lengths = [430, 1, 0, 811, ps * 9, 250]
    B = len(lengths)
    rng = np.random.default_rng(53)
    labels = [np.sort(rng.integers(0, 7, n)).astype(np.uint8) for n in lengths]
    kv = [[to_dev(x) for x in synth.kv_host(53, b, L, Hkv, 0, n, labels[b])] for b, n in enumerate(lengths)]
    new = [np.where(rng.random(B) < 0.3, rng.integers(1, 7, B), 6).astype(np.uint8) for _ in range(steps)]
    x = [[to_dev(t) for t in (synth.q_host(53, B, L, Hq, Hkv, s + 1), *synth.step_kv_host(
        53, [n + s for n in lengths], new[s], L, Hkv))] for s in range(steps)]
    rows = [[[t[:, l].contiguous() for t in x[s]] for l in range(L)] for s in range(steps)]
    budget = np.array([max(1, (n + ps - 1) // ps - 3) for n in lengths], np.int32)
    got = []
    for wait in (False, True):
        c = md.Cache(L, Hq, Hkv, ps, B, 100, 100 * B, region_aligned_pages=aligned)
        if kernel == "persistent":
            c.debug_set(md.MD_DEBUG_GRID_LIMIT, 512)
        elif kernel != "by cost":
            c.debug_set(md.MD_DEBUG_CLUSTER_FORM, 1 + 256 * 8 if kernel == "8 warps" else 2 + 256 * 4 + 65536)
        for r in range(7):
            c.set_region_params(r, 1.0 - 0.1 * r, 20.0, r == 0)
        for b in range(B):
            if lengths[b]:
                c.append_tokens(b, labels[b], *kv[b])
        out = torch.zeros((steps, L, B, Hq, 128), dtype=torch.int16, device="cuda")
        whole = torch.zeros((steps, B, L, Hq, 128), dtype=torch.int16, device="cuda")
        masses = []
        torch.cuda.synchronize()
        for s in range(steps):
            if s % 4 == 3:
                c.decode_step(B, *x[s], new[s], whole[s])
            else:
                for l in range(L):
                    c.decode_layer(l, B, *rows[s][l], new[s], out[s, l])
                    if wait:
                        torch.cuda.synchronize()
            if wait:
                torch.cuda.synchronize()
            masses.append(c.get_state(md.MD_STATE_MASS))
            if (s + 1) % window == 0:
                c.evict(budget)
                if wait:
                    torch.cuda.synchronize()
        assert c.sync() == md.MD_OK
        used = torch.cat([c.get_state(md.MD_STATE_BLOCK_TABLE)[b, :c.query(md.MD_QUERY_PAGES, b)] for b in range(B)])
        got.append([out, whole, *masses, *[c.get_state(k) for k in (
            md.MD_STATE_BLOCK_TABLE, md.MD_STATE_FREE, md.MD_STATE_PAGE_FILL, md.MD_STATE_SEQ_TOKENS)]] +
            [c.get_state(k).view(-1, ps)[used.long()] for k in (
                md.MD_STATE_REGION, md.MD_STATE_A, md.MD_STATE_T_REF, md.MD_STATE_AHAT)])
        c.close()
    for i, (a, b) in enumerate(zip(*got)):
        assert torch.equal(a, b), i


@pytest.mark.parametrize("n", [40, 900])
def test_output_at_any_address(n):
    """The output may start at any 2-byte address: the wide stores are taken
    only where it is aligned for them."""
    w = synth.custom_workload("addr", L=1, Hq=16, Hkv=2, page_size=16, lengths=[n], budget_frac=1.0, steps=1, seed=43)
    outs = []
    for shift in (0, 1, 4):
        c = md.Cache(1, 16, 2, 16, 1, 80, 80)
        k, v = synth.kv_host(w.seed, 0, 1, 2, 0, n, w.regions[0])
        c.append_tokens(0, w.regions[0], to_dev(k), to_dev(v))
        kn, vn = synth.step_kv_host(w.seed, [n], [6], 1, 2)
        buf = torch.zeros(16 * 128 + 8, dtype=torch.int16, device="cuda")
        c.decode_step(1, to_dev(synth.q_host(w.seed, 1, 1, 16, 2, 1)), to_dev(kn), to_dev(vn), [6],
                      buf.data_ptr() + 2 * shift)
        assert c.sync() == md.MD_OK
        assert int(buf[:shift].abs().sum()) == 0 and int(buf[shift + 16 * 128:].abs().sum()) == 0
        outs.append(buf[shift:shift + 16 * 128].clone())
        c.close()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


@pytest.mark.parametrize("ps,aligned,reduce", [(16, 0, 0), (32, 0, 1), (16, 1, 1), (32, 1, 0)])
def test_one_launch_observation_selects_what_the_two_kernels_select(ps, aligned, reduce):
    """A batch of short sequences, scored and selected in one launch, against
    the same batch with the calibration histogram on, which takes the two
    kernels: token state, page scores, tables, fills, counts and evicted pages
    bit for bit.  Pages at the ends of warps and of the kernel's range (256
    pages, 4,096 slots), none, one, several and all evictable pages evicted,
    equal scores (b = 0 and no attention weight)."""
    run = 3 * ps - 5 if aligned else 23       # tokens per label: aligned, 3 pages each, the third not full
    sizes = [1, ps, 31 * ps, 32 * ps, 33 * ps - 1, 4096 // ps * ps - 2, 70 * ps + 5, 5 * ps]
    if aligned:                               # the new token (label 6) opens the last page of the range
        sizes = [1, ps, 10 * run, 10 * run + 2 * ps, 11 * run - 1, 85 * run if ps == 16 else 42 * run + 10, 23 * run + 5,
                 2 * run]
    cut = [0, 1, 1, 31, 17, 90, 200, 99]
    B = len(sizes)
    for weight in (1.0, 0.0):
        got = []
        for two_kernels in (False, True):
            c = md.Cache(1, 4, 1, ps, B, 700, 700 * B, page_reduce=reduce, attn_weight=weight,
                         region_aligned_pages=aligned)
            for r in range(7):
                c.set_region_params(r, 0.0 if weight == 0.0 else 0.3 + 0.1 * r, 20.0, r == 0)
            for b, m in enumerate(sizes):
                lab = (np.arange(m) // run % 7).astype(np.uint8)
                k, v = synth.kv_host(19, b, 1, 1, 0, m, lab)
                c.append_tokens(b, lab, to_dev(k), to_dev(v), -(np.arange(m, dtype=np.int32)[::-1] // 40))
            c.calib_enable(two_kernels)
            q = synth.q_host(19, B, 1, 4, 1, 1)
            kn, vn = synth.step_kv_host(19, sizes, [6] * B, 1, 1)
            out = torch.empty((B, 1, 4, 128), dtype=torch.int16, device="cuda")
            c.decode_step(B, to_dev(q), to_dev(kn), to_dev(vn), [6] * B, out)
            pages = [c.query(md.MD_QUERY_PAGES, b) for b in range(B)]
            assert max(pages) == 4096 // ps
            ids = torch.full((B, 700), -7, dtype=torch.int32, device="cuda")
            before = c.get_state(md.MD_STATE_BLOCK_TABLE)
            c.profile_enable(True)
            st, n_ev = c.evict([max(0, p - e) for p, e in zip(pages, cut)], ids)
            ran = c.profile_read()
            assert (ran["score"][1], ran["select"][1]) == (1, int(two_kernels))
            assert c.sync() == md.MD_OK
            got.append([before, torch.from_numpy(n_ev), ids] + [c.get_state(w) for w in (
                md.MD_STATE_PAGE_SCORE, md.MD_STATE_BLOCK_TABLE, md.MD_STATE_PAGE_FILL, md.MD_STATE_SEQ_TOKENS)])
            slot = before.cpu().numpy()
            slot = torch.from_numpy(np.concatenate([slot[b, :pages[b]] for b in range(B)]).astype(np.int64)).cuda()
            got[-1] += [c.get_state(w).view(-1, ps)[slot] for w in (
                md.MD_STATE_A, md.MD_STATE_T_REF, md.MD_STATE_AHAT, md.MD_STATE_TOKEN_PRIO, md.MD_STATE_WINDOW)]
            c.close()
        assert int(got[0][1].sum()) > 100
        for x, y in zip(*got):
            assert torch.equal(x, y)


@pytest.mark.parametrize("ps,aligned", [(16, 0), (32, 0), (16, 1), (32, 1)])
@pytest.mark.parametrize("runs", ["spans", "single tokens"])
def test_append_in_one_call_and_in_pieces(ps, aligned, runs):
    """The same tokens appended in one call and in pieces of odd sizes leave
    the same pool, token state and page tables, bit for bit, with few runs of
    equal labels and steps (passed in the launch parameters) and with more than
    fit there (passed through the workspace)."""
    L, Hkv, n = 2, 3, 1333
    rng = np.random.default_rng(11)
    lab = np.repeat(rng.integers(0, 7, 40), 34)[:n].astype(np.uint8) if runs == "spans" else \
        (np.arange(n) * 5 % 7).astype(np.uint8)
    step = -(np.arange(n, dtype=np.int32)[::-1] // 100) if runs == "spans" else -np.arange(n, dtype=np.int32) % 50 - 49
    k, v = synth.kv_host(13, 0, L, Hkv, 0, n, lab)
    kd, vd = to_dev(k), to_dev(v)
    states = []
    for sizes in ([n], [1, 15, 16, 17, 31, 33, 5, 700, 64, n]):
        c = md.Cache(L, 6, Hkv, ps, 2, n, n + 4, region_aligned_pages=aligned)
        c.set_region_params(0, 1.0, 10.0, True)
        i = 0
        for m in sizes:
            m = min(m, n - i)
            c.append_tokens(1, lab[i:i + m], kd[:, :, i:i + m].contiguous(), vd[:, :, i:i + m].contiguous(), step[i:i + m])
            i += m
        assert c.query(md.MD_QUERY_TOKENS, 1) == n
        states.append([c.get_state(w) for w in (
            md.MD_STATE_POOL, md.MD_STATE_REGION, md.MD_STATE_T_INS, md.MD_STATE_T_REF, md.MD_STATE_A,
            md.MD_STATE_BLOCK_TABLE, md.MD_STATE_PAGE_FILL, md.MD_STATE_SEQ_TOKENS)] +
            [torch.tensor([c.query(q, 1) for q in (md.MD_QUERY_PAGES, md.MD_QUERY_PINNED_PAGES, md.MD_QUERY_FREE_TOP)])])
        slots = c.get_state(md.MD_STATE_BLOCK_TABLE)[1].cpu().numpy()
        if not aligned:      # and the pool holds the tokens where the table says
            at = torch.from_numpy(slots[np.arange(n) // ps] * ps + np.arange(n) % ps).cuda().long()
            pool = c.get_state(md.MD_STATE_POOL)
            got = pool[:, :, :, 0].permute(0, 2, 1, 3, 4).reshape(L, Hkv, -1, 128)[:, :, at]
            assert torch.equal(got, kd)
            assert torch.equal(c.get_state(md.MD_STATE_REGION)[at].cpu(), torch.from_numpy(lab))
            assert torch.equal(c.get_state(md.MD_STATE_T_INS)[at].cpu(), torch.from_numpy(step))
        c.close()
    for x, y in zip(*states):
        assert torch.equal(x, y)


@pytest.mark.parametrize("ps,aligned", [(16, 0), (32, 0), (16, 1), (32, 1)])
@pytest.mark.parametrize("entry", ["device", "layers"])
@pytest.mark.parametrize("kernel", ["cluster", "persistent", "persistent, many items"])
def test_append_inside_attention_writes_what_the_append_kernel_writes(ps, aligned, entry, kernel):
    """Decode steps whose attention launch appends the new tokens (the cluster
    kernel; the persistent one with contiguous pages and few items per CTA, else
    it follows an append launch) leave the same pool, token state and
    page tables, bit for bit, as steps with host buffers, whose append is always
    a launch of its own.  Lengths put the new token on the first and the last
    slot of a page, on both 16-token tiles of a 32-token page and into an empty
    sequence; region changes open pages early."""
    L, Hq, Hkv = 2, 16, 2
    lengths = [0, 1, ps - 1, ps, ps + 1, 5 * ps - 1, 33 * ps, 700]
    if kernel == "persistent, many items":                          # 4,000 items of the step, 500 of a layer
        L, lengths = 8, lengths + [3 * i % 67 for i in range(242)]
    B = len(lengths)
    rng = np.random.default_rng(7)
    pages = sum(n // ps + (40 if aligned else 12) for n in lengths) + 100
    caches = [md.Cache(L, Hq, Hkv, ps, B, 64, pages, region_aligned_pages=aligned) for _ in range(2)]
    if kernel != "cluster":
        for c in caches:
            c.debug_set(md.MD_DEBUG_GRID_LIMIT, 128)
    regs = [np.sort(rng.integers(0, 7, n)).astype(np.uint8) for n in lengths]
    for c in caches:
        for r in range(7):
            c.set_region_params(r, 1.0, 50.0, r == 0)
        for b, n in enumerate(lengths):
            if n:
                k, v = synth.kv_host(3, b, L, Hkv, 0, n, regs[b])
                c.append_tokens(b, regs[b], to_dev(k), to_dev(v))
    for step in range(ps + 2):
        new = rng.integers(0, 7, B).astype(np.uint8) if step % 3 == 0 else np.full(B, 6, np.uint8)
        q = synth.q_host(3, B, L, Hq, Hkv, step + 1)
        kn, vn = synth.step_kv_host(3, [n + step for n in lengths], new, L, Hkv)
        out = torch.empty((B, L, Hq, 128), dtype=torch.int16, device="cuda")
        if entry == "device":
            caches[0].decode_step(B, to_dev(q), to_dev(kn), to_dev(vn), new, out)
        else:
            for l in range(L):
                o = torch.empty((B, Hq, 128), dtype=torch.int16, device="cuda")
                caches[0].decode_layer(l, B, to_dev(q[:, l]), to_dev(kn[:, l]), to_dev(vn[:, l]), new, o)
                out[:, l] = o
        pin = [torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).pin_memory() for a in (q, kn, vn)]
        out_h = torch.empty((B, L, Hq, 128), dtype=torch.int16).pin_memory()
        caches[1].decode_step_host(B, *pin, new, out_h)
        assert caches[1].sync() == md.MD_OK
        diff = synth.bf16_to_f64(out.cpu().numpy().view(np.uint16)) - synth.bf16_to_f64(out_h.numpy().view(np.uint16))
        assert np.max(np.abs(diff)) <= TOL_O_ABS
        if step % 5 == 4:      # an eviction in between: pages are freed and taken again
            for c in caches:
                c.evict([max(2, c.query(md.MD_QUERY_PAGES, b) - 2) for b in range(B)])
        for what in (md.MD_STATE_POOL, md.MD_STATE_REGION, md.MD_STATE_T_INS, md.MD_STATE_BLOCK_TABLE,
                     md.MD_STATE_PAGE_FILL, md.MD_STATE_SEQ_TOKENS, md.MD_STATE_FREE):
            assert torch.equal(caches[0].get_state(what), caches[1].get_state(what)), (step, what)
    for c in caches:
        c.close()


@pytest.mark.parametrize("ps,aligned,persistent", [(16, 0, 0), (32, 0, 0), (32, 1, 0), (16, 0, 1), (32, 0, 1),
                                                   (16, 1, 1), (32, 1, 1)])
@pytest.mark.parametrize("entry", ["device", "host"])
def test_recycled_pages_leave_nothing_in_the_output(ps, aligned, persistent, entry):
    """Pages that an evicted sequence with infinite and NaN values leaves behind
    give the next sequence the same output and masses, bit for bit, as pages
    never used: what a slot past a page's tokens holds must not reach them."""
    L, Hq, Hkv, n = 2, 16, 2, 3 * 101 + 1
    lab = (np.arange(n) // 101 % 7).astype(np.uint8)       # aligned: partly filled pages inside
    k, v = (to_dev(x) for x in synth.kv_host(37, 0, L, Hkv, 0, n, lab))
    bad = torch.full_like(v, 0x7F80)
    bad[:, :, ::3] = 0x7FFF
    q = synth.q_host(37, 1, L, Hq, Hkv, 1)
    kn, vn = synth.step_kv_host(37, [n], [lab[-1]], L, Hkv)
    got = []
    for used in (False, True):
        c = md.Cache(L, Hq, Hkv, ps, 2, 64, 64, region_aligned_pages=aligned)
        if persistent:
            c.debug_set(md.MD_DEBUG_GRID_LIMIT, 128)
        if used:
            for part in (slice(0, 150), slice(150, n)):
                c.append_tokens(1, np.full(part.stop - part.start, 6, np.uint8), k[:, :, part].contiguous(),
                                bad[:, :, part].contiguous())
            st, n_ev = c.evict([0, 0])
            assert st == md.MD_WARN_OVER_BUDGET and n_ev[1] == (n + ps - 1) // ps - 1
        c.append_tokens(0, lab, k, v)
        slots = c.get_state(md.MD_STATE_BLOCK_TABLE)[0, :c.query(md.MD_QUERY_PAGES, 0)].long()
        if entry == "device":
            out = torch.empty((1, L, Hq, 128), dtype=torch.int16, device="cuda")
            c.decode_step(1, to_dev(q), to_dev(kn), to_dev(vn), [lab[-1]], out)
        else:
            pin = [torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).pin_memory() for a in (q, kn, vn)]
            out = torch.empty((1, L, Hq, 128), dtype=torch.int16).pin_memory()
            c.decode_step_host(1, *pin, [lab[-1]], out)
        assert c.sync() == md.MD_OK
        got.append((out.cpu(), c.get_state(md.MD_STATE_MASS).view(-1, ps)[slots]))
        c.close()
    assert torch.isfinite(got[1][0].view(torch.bfloat16).float()).all()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


def test_argument_forms_give_the_same_step():
    """Labels and budgets as exact arrays (taken in place), lists, other
    integer types and strided arrays; host buffers as tensors and as numpy
    arrays: the same outputs and counts."""
    L, Hq, Hkv, ps, n = 2, 8, 2, 16, [100, 333]
    q = synth.q_host(23, 2, L, Hq, Hkv, 1)
    kn, vn = synth.step_kv_host(23, n, [5, 6], L, Hkv)
    forms = [np.array([5, 6], np.uint8), [5, 6], np.array([5, 6], np.int64), np.array([5, 9, 6, 9], np.uint8)[::2]]
    cuts = [np.array([4, 9], np.int32), [4, 9], np.array([4, 9], np.int64), np.array([4, 0, 9, 0], np.int32)[::2]]
    seen = []
    for entry in ("device", "layers", "host tensors", "host arrays"):
        for regs, cut in zip(forms, cuts):
            c = md.Cache(L, Hq, Hkv, ps, 2, 30, 60)
            for b, m in enumerate(n):
                k, v = synth.kv_host(23, b, L, Hkv, 0, m)
                c.append_tokens(b, np.full(m, 4, np.uint8), to_dev(k), to_dev(v))
            out = torch.empty((2, L, Hq, 128), dtype=torch.int16, device="cuda")
            if entry == "device":
                c.decode_step(2, to_dev(q), to_dev(kn), to_dev(vn), regs, out)
            elif entry == "layers":
                for l in range(L):
                    o = torch.empty((2, Hq, 128), dtype=torch.int16, device="cuda")
                    c.decode_layer(l, 2, to_dev(q[:, l]), to_dev(kn[:, l]), to_dev(vn[:, l]), regs, o)
                    out[:, l] = o
            else:
                host = [np.ascontiguousarray(a).view(np.int16) for a in (q, kn, vn)]
                res = np.zeros((2, L, Hq, 128), np.int16)
                if entry == "host tensors":
                    c.decode_step_host(2, *[torch.from_numpy(a) for a in host], regs, torch.from_numpy(res))
                else:
                    c.decode_step_host(2, *host, regs, res)
                assert c.sync() == md.MD_OK
                out = torch.from_numpy(res).cuda()
            st, n_ev = c.evict(cut)
            assert st == md.MD_OK and n_ev.dtype == np.int32 and list(n_ev) == [3, 12]
            seen.append((out.clone(), c.get_state(md.MD_STATE_REGION), c.get_state(md.MD_STATE_BLOCK_TABLE)))
            with pytest.raises(md.MemDecayError):
                c.decode_step(3, 1, 1, 1, regs, 1)
            c.close()
    x = synth.bf16_to_f64(seen[0][0].cpu().numpy().view(np.uint16))
    for o, reg, tab in seen[1:]:
        y = synth.bf16_to_f64(o.cpu().numpy().view(np.uint16))
        assert np.max(np.abs(x - y)) <= TOL_O_ABS
        assert torch.equal(reg, seen[0][1]) and torch.equal(tab, seen[0][2])


@pytest.mark.parametrize("pages", [1, 3, 4097])
def test_state_copies_at_any_address(pages):
    """Every state array reads back the same into an aligned buffer (copied by
    a kernel where it is small) and into one that is not aligned for that."""
    c = md.Cache(1, 4, 1, 16, 2, pages, pages)
    k, v = synth.kv_host(29, 0, 1, 1, 0, 16)
    c.append_tokens(1, np.arange(16) % 7, to_dev(k), to_dev(v), -np.arange(16))
    for what in range(15):
        a = c.get_state(what)
        raw = a.contiguous().view(torch.uint8).view(-1)
        buf = torch.zeros(raw.numel() + 32, dtype=torch.uint8, device="cuda")
        off = 1 if a.element_size() == 1 else a.element_size()
        assert md.lib().md_get_state(c.h, what, buf.data_ptr() + off, raw.numel()) == md.MD_OK
        assert torch.equal(buf[off:off + raw.numel()], raw), what
        assert int(buf[:off].sum()) == 0 and int(buf[off + raw.numel():].sum()) == 0, what
    c.close()


def test_checkpoint_restore_replays_step():
    w = synth.custom_workload("ckpt", L=2, Hq=8, Hkv=2, page_size=16, lengths=[900],
                              budget_frac=0.3, steps=2, seed=9)
    ls = Lockstep(w)
    ls.prefill()
    ls.decode()
    ls.observe()
    saved = ls.gpu.save_state()
    q = synth.q_host(w.seed, 1, w.L, w.Hq, w.Hkv, 99)
    kn, vn = synth.step_kv_host(w.seed, [5000], [6], w.L, w.Hkv)
    res = []
    for _ in range(2):
        ls.gpu.load_state(saved)
        out = torch.empty((1, w.L, w.Hq, 128), dtype=torch.int16, device="cuda")
        ls.gpu.decode_step(1, to_dev(q), to_dev(kn), to_dev(vn), [6], out)
        ls.gpu.evict([3])
        res.append((out.clone(), ls.gpu.get_state(md.MD_STATE_BLOCK_TABLE),
                    ls.gpu.get_state(md.MD_STATE_PAGE_SCORE)))
    torch.cuda.synchronize()
    for x, y in zip(res[0], res[1]):
        assert torch.equal(x, y)


def test_checkpoint_carries_the_calibration_histogram():
    """A checkpoint taken with calibration on restores the histogram (and the
    switch): replaying a step from it gives the same histogram as the first
    time, whatever was gathered in between."""
    w = synth.custom_workload("ckcal", L=2, Hq=8, Hkv=2, page_size=16, lengths=[900, 400],
                              budget_frac=0.4, steps=4, seed=13, structured=True)
    ls = Lockstep(w)
    ls.prefill()
    ls.gpu.calib_enable(True)
    ls.decode()
    ls.observe()
    saved = ls.gpu.save_state()
    q = synth.q_host(w.seed, w.B, w.L, w.Hq, w.Hkv, 7, True)
    kn, vn = synth.step_kv_host(w.seed, [5000, 5000], [6, 6], w.L, w.Hkv, True)
    res = []
    for _ in range(2):
        ls.gpu.load_state(saved)
        out = torch.empty((w.B, w.L, w.Hq, 128), dtype=torch.int16, device="cuda")
        ls.gpu.decode_step(w.B, to_dev(q), to_dev(kn), to_dev(vn), [6, 6], out)
        ls.gpu.evict(w.budget_pages)
        s, n = ls.gpu.calib_read()
        res.append((np.array(s), np.array(n)))
        # gather more in between: the restore must undo it
        ls.gpu.decode_step(w.B, to_dev(q), to_dev(kn), to_dev(vn), [6, 6], out)
        ls.gpu.evict(w.budget_pages)
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])
    assert res[0][1].sum() > 0


def test_partial_batch_leaves_the_other_sequences_untouched():
    """Steps over sequences [0, batch) with batch < max_batch: the covered
    sequences follow the oracle run with the same batch (outputs, evictions,
    block tables), and the uncovered one keeps its block-table row, token
    count and per-token state bit for bit."""
    w = synth.custom_workload("part", L=2, Hq=16, Hkv=2, page_size=16, lengths=[800, 1300, 600],
                              budget_frac=0.4, steps=3, seed=17, structured=True)
    ls = Lockstep(w)
    ls.prefill()
    B, ps = 2, w.page_size
    bt0 = ls.gpu.get_state(md.MD_STATE_BLOCK_TABLE).cpu().numpy()
    n2 = ls.gpu.query(md.MD_QUERY_TOKENS, 2)
    slots2 = np.array([bt0[2, i // ps] * ps + i % ps for i in range(n2)])
    state = lambda: [ls.gpu.get_state(x).cpu().numpy()[slots2] for x in
                     (md.MD_STATE_A, md.MD_STATE_T_REF, md.MD_STATE_REGION, md.MD_STATE_WINDOW)]
    s0 = state()
    for t in range(1, 4):
        q = synth.q_host(w.seed, B, w.L, w.Hq, w.Hkv, t, True)
        kn, vn = synth.step_kv_host(w.seed, ls.pos[:B], [6] * B, w.L, w.Hkv, True)
        out = torch.empty((B, w.L, w.Hq, 128), dtype=torch.int16, device="cuda")
        ls.gpu.decode_step(B, to_dev(q), to_dev(kn), to_dev(vn), [6] * B, out)
        O = ls.orc.decode_step(B, q, kn, vn, [6] * B)
        for b in range(B):
            ls.pos[b] += 1
        err = float(np.max(np.abs(synth.bf16_to_f64(out.cpu().numpy().view(np.uint16)) - O)))
        assert err <= TOL_O_ABS, (t, err)
        st, n_ev = ls.gpu.evict(w.budget_pages[:B])
        _, n_ev_o, _, _ = ls.orc.evict(B, w.budget_pages[:B])
        assert list(n_ev) == list(n_ev_o), t
        bt = ls.gpu.get_state(md.MD_STATE_BLOCK_TABLE).cpu().numpy()
        for b in range(B):
            assert list(bt[b, :len(ls.orc.block[b])]) == list(ls.orc.block[b]), (t, b)
        assert np.array_equal(bt[2], bt0[2]), t
    assert ls.gpu.query(md.MD_QUERY_TOKENS, 2) == n2
    for x, y in zip(state(), s0):
        assert np.array_equal(x, y)
    assert ls.gpu.sync() == md.MD_OK


def test_capacity_and_argument_errors_are_synchronous():
    c = md.Cache(1, 8, 2, 16, 2, 4, 6)
    k = torch.zeros((1, 2, 80, 128), dtype=torch.int16, device="cuda")
    with pytest.raises(md.MemDecayError) as e:
        c.append_tokens(0, np.zeros(80, np.uint8), k, k)          # 5 pages > 4
    assert e.value.status == md.MD_ERR_CAPACITY
    assert c.query(md.MD_QUERY_TOKENS, 0) == 0 and c.query(md.MD_QUERY_FREE_TOP) == 6
    with pytest.raises(md.MemDecayError) as e:
        c.append_tokens(0, np.full(3, 9, np.uint8), k[:, :, :3].contiguous(), k[:, :, :3].contiguous())
    assert e.value.status == md.MD_ERR_INVALID_ARG
    with pytest.raises(md.MemDecayError) as e:
        c.append_tokens(0, np.zeros(3, np.uint8), k, k, insert_steps=[0, 1, 5])
    assert e.value.status == md.MD_ERR_INVALID_ARG
    with pytest.raises(md.MemDecayError) as e:
        c.set_region_params(1, 1.0, 0.0, False)
    assert e.value.status == md.MD_ERR_INVALID_ARG
    c.append_tokens(0, np.zeros(3, np.uint8), k[:, :, :3].contiguous(), k[:, :, :3].contiguous())
    with pytest.raises(md.MemDecayError) as e:
        c.set_region_params(0, 1.0, 10.0, True)   # pinned flag with tokens cached
    assert e.value.status == md.MD_ERR_STATE
    for key, bad in ((md.MD_DEBUG_ZERO_COPY, 2), (md.MD_DEBUG_COMBINE_OVERHEAD, -1),
                     (md.MD_DEBUG_COMBINE_OVERHEAD, 1 << 20), (md.MD_DEBUG_GRID_LIMIT, md.MD_MAX_CHUNKS - 1),
                     (md.MD_DEBUG_FORCE_CHUNKS, md.MD_MAX_CHUNKS + 1), (md.MD_DEBUG_CLUSTER_FORM, 3 + 256 * 4),
                     (md.MD_DEBUG_CLUSTER_FORM, 32 + 256 * 4), (md.MD_DEBUG_CLUSTER_FORM, 2 + 256 * 5),
                     (md.MD_DEBUG_CLUSTER_FORM, 2 + 256 * 4 + 65536 * 2), (md.MD_DEBUG_CLUSTER_FORM, -1), (99, 0)):
        with pytest.raises(md.MemDecayError) as e:
            c.debug_set(key, bad)
        assert e.value.status == md.MD_ERR_INVALID_ARG, (key, bad)
    assert c.sync() == md.MD_OK


def test_single_token_and_no_eviction_edges():
    """One cached token (o = v exactly, Abar = 1), and budgets at or above
    the page count (nothing evicted)."""
    w = synth.custom_workload("tiny", L=1, Hq=8, Hkv=2, page_size=16, lengths=[0],
                              budget_frac=1.0, steps=48, seed=10)
    ls = Lockstep(w)
    ls.decode()
    n = ls.observe(budgets=[5])
    assert list(n) == [0]
    ah = ls.gpu.get_state(md.MD_STATE_AHAT).cpu().numpy()
    slot = ls.orc.slots(0)[0]
    assert abs(ah[slot] - 1.0) < 1e-6
    for _ in range(40):
        ls.decode()
        ls.observe(budgets=[100])
    ls.check_layout()


def test_maximum_batch_of_ragged_sequences():
    """MD_MAX_BATCH sequences in one handle, ragged from empty (the first token
    arrives with the first decode step) to several pages with a partial last
    page: every sequence checked at every step."""
    lengths = [0 if i % 97 == 0 else 1 + (37 * i) % 400 for i in range(md.MD_MAX_BATCH)]
    w = synth.custom_workload("maxbatch", L=1, Hq=8, Hkv=2, page_size=16, lengths=lengths,
                              budget_frac=0.5, steps=3, seed=12)
    ls = Lockstep(w).run()
    ls.check_layout()


def test_longest_sequence_the_chunking_allows():
    """One sequence at the block-table limit, MD_MAX_CHUNKS chunks of
    MD_MAX_CHUNK_TOKENS tokens (8,192 pages of 32) once the decode step's token
    is appended, then evicted to 5% of its pages."""
    limit = md.MD_MAX_CHUNKS * md.MD_MAX_CHUNK_TOKENS
    w = synth.custom_workload("maxlen", L=1, Hq=8, Hkv=2, page_size=32, lengths=[limit - 1],
                              budget_frac=0.05, steps=3, seed=13)
    ls = Lockstep(w, p_max=limit // 32).run()
    ls.check_layout()


def test_device_wait_timeout_is_reported_not_hung():
    """An exchange wait that nothing completes (an injected extra arrival)
    runs out after its bounded spin; the kernel records the timeout and
    returns; the CUDA context stays usable and the handle refuses more work."""
    w = synth.custom_workload("to", L=1, Hq=8, Hkv=2, page_size=16, lengths=[600],
                              budget_frac=0.5, steps=1, seed=11)
    ls = Lockstep(w)
    ls.prefill()
    ls.gpu.debug_set(md.MD_DEBUG_SPIN_LIMIT_NS, 20_000_000)
    ls.gpu.debug_set(md.MD_DEBUG_EXTRA_ARRIVALS, 1)
    q = synth.q_host(w.seed, 1, 1, 8, 2, 1)
    kn, vn = synth.step_kv_host(w.seed, [600], [6], 1, 2)
    out = torch.empty((1, 1, 8, 128), dtype=torch.int16, device="cuda")
    ls.gpu.decode_step(1, to_dev(q), to_dev(kn), to_dev(vn), [6], out)
    assert ls.gpu.sync() == md.MD_ERR_DEVICE_TIMEOUT
    with pytest.raises(md.MemDecayError) as e:
        ls.gpu.evict([2])
    assert e.value.status == md.MD_ERR_STATE
    x = torch.arange(10, device="cuda").sum()
    assert int(x) == 45
    ls2 = Lockstep(w)
    ls2.prefill()
    ls2.decode()
    ls2.observe()


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("n", [600, 6000])
def test_wait_limit_shorter_than_a_copy(persistent, n):
    """With the smallest wait limit (1 us, less than a copy from HBM may take)
    a step either finishes or reports the timeout, its copies have landed before
    the kernel ends, and a new handle over the same memory computes as ever."""
    w = synth.custom_workload("short", L=2, Hq=16, Hkv=2, page_size=16, lengths=[n, 300], budget_frac=0.5, steps=2,
                              seed=51)
    for _ in range(4):
        ls = Lockstep(w)
        ls.prefill()
        ls.gpu.debug_set(md.MD_DEBUG_SPIN_LIMIT_NS, 1000)
        if persistent:
            ls.gpu.debug_set(md.MD_DEBUG_GRID_LIMIT, 128)
        q = synth.q_host(w.seed, 2, 2, 16, 2, 1)
        kn, vn = synth.step_kv_host(w.seed, ls.pos, [6, 6], 2, 2)
        out = torch.empty((2, 2, 16, 128), dtype=torch.int16, device="cuda")
        ls.gpu.decode_step(2, to_dev(q), to_dev(kn), to_dev(vn), [6, 6], out)
        assert ls.gpu.sync() in (md.MD_OK, md.MD_ERR_DEVICE_TIMEOUT)
        ls.gpu.close()
    Lockstep(w).run().check_layout()
