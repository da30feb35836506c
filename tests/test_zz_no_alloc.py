"""md_attend_mass_noalloc: stage 1 for callers that cannot allocate device
memory (a serving engine that owns the allocator, code that must not
allocate once it is running, a fixed memory budget).  It uses a fixed
scratch array inside the library instead of a workspace.  Its output must
match the workspace path (md_decode_step's attention output, and its step
mass per token: the sum of the rows over layers and KV heads)
within the parity tolerances, on two calls in a row (the second call finds
the first call's leftovers in the shared array)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2607_10582_gb300 as md  # noqa: E402
import synth  # noqa: E402
from paper_2607_10582_gb300 import build as mdbuild  # noqa: E402
from tests.attention_shapes import NOALLOC_PERSISTENT  # noqa: E402
from tests.gpu_harness import TOL_FLOOR, TOL_O_ABS, TOL_REL, to_dev  # noqa: E402

mdbuild.build()
synth.build()


@pytest.mark.parametrize("L,Hq,ps,lengths", [
    (2, 16, 16, [900, 2500]),
    (2, 12, 32, [3000, 70, 1500]),
    # many items and long sequences, one short one: clusters of 8-warp CTAs
    (16, 16, 16, [3000] * 7 + [40] + [3000] * 8),
    # a serving batch shaped like the 3B geometry at budget: one CTA per item
    (36, 16, 16, [420 + 9 * i for i in range(32)]),
])
def test_noalloc_matches_workspace_path_twice(L, Hq, ps, lengths):
    w = synth.custom_workload("noalloc", L=L, Hq=Hq, Hkv=2, page_size=ps, lengths=lengths,
                              budget_frac=0.5, steps=4, seed=21, structured=True)
    B, L, Hkv, D = w.B, w.L, w.Hkv, 128
    c = md.Cache(L, Hq, Hkv, ps, B, w.max_pages_per_seq(), w.num_phys_pages())
    for r in range(7):
        c.set_region_params(r, w.base[r], w.half_life[r], bool(w.pinned[r]))
    for b in range(B):
        k, v = synth.kv_host(w.seed, b, L, Hkv, 0, w.n0(b), w.regions[b], True)
        c.append_tokens(b, w.regions[b], to_dev(k), to_dev(v))
    q = to_dev(synth.q_host(w.seed, B, L, Hq, Hkv, 1, True))
    kn, vn = synth.step_kv_host(w.seed, [w.n0(b) for b in range(B)], [6] * B, L, Hkv, True)
    out_ref = torch.empty((B, L, Hq, D), dtype=torch.int16, device="cuda")
    c.decode_step(B, q, to_dev(kn), to_dev(vn), [6] * B, out_ref)
    mass_ref = c.get_state(md.MD_STATE_MASS)
    pool = c.get_state(md.MD_STATE_POOL)
    bt = c.get_state(md.MD_STATE_BLOCK_TABLE)
    n_tok = np.array([c.query(md.MD_QUERY_TOKENS, b) for b in range(B)], np.int32)
    torch.cuda.synchronize()

    bt_h = bt.cpu().numpy()
    slots = np.concatenate([[bt_h[b, i // ps] * ps + i % ps for i in range(n_tok[b])] for b in range(B)])
    ref_o = synth.bf16_to_f64(out_ref.cpu().numpy().view(np.uint16))
    # the workspace path keeps the step's mass per token, summed over layers
    # and query heads, in fixed point (2^48 = 1.0)
    ref_m = mass_ref.cpu().numpy()[slots].astype(np.float64) * 2.0 ** -48
    stream = torch.cuda.current_stream().cuda_stream
    for call in range(2):
        out = torch.zeros_like(out_ref)
        mass = torch.zeros((L * Hkv, c.P_phys * ps), dtype=torch.float32, device="cuda")
        st = md.lib().md_attend_mass_noalloc(pool.data_ptr(), bt.data_ptr(), n_tok.ctypes.data, q.data_ptr(),
                                             out.data_ptr(), mass.data_ptr(), B, L, Hq, Hkv, ps,
                                             c.P_max, c.P_phys, stream)
        assert st == md.MD_OK, (call, st)
        torch.cuda.synchronize()
        got_o = synth.bf16_to_f64(out.cpu().numpy().view(np.uint16))
        assert np.max(np.abs(got_o - ref_o)) <= TOL_O_ABS, call
        got_m = mass.cpu().numpy()[:, slots].astype(np.float64).sum(axis=0)
        rel = np.max(np.abs(got_m - ref_m) / (np.abs(ref_m) + TOL_FLOOR))
        assert rel <= TOL_REL, (call, rel)
    c.close()


@pytest.mark.parametrize("L,Hq,Hkv,ps,lengths", NOALLOC_PERSISTENT)
def test_noalloc_on_the_persistent_kernel_twice(L, Hq, Hkv, ps, lengths):
    """The persistent kernel with the fixed array (score rows, counters, and
    partials where an item has several chunks) against attention in 64 bits, on
    two calls in a row: the second finds the first one's leftovers."""
    B, P, G = len(lengths), max(lengths) // ps + 1, Hq // Hkv
    pages = [(n + ps - 1) // ps for n in lengths]
    NP = sum(pages)
    g = torch.Generator(device="cuda").manual_seed(59)
    pool = torch.randn((L, NP, Hkv, 2, ps, 128), generator=g, device="cuda").bfloat16()
    ids = torch.randperm(NP, generator=g, device="cuda")
    bt = torch.zeros((B, P), dtype=torch.int32, device="cuda")
    first = 0
    for b in range(B):
        bt[b, :pages[b]] = ids[first:first + pages[b]]
        first += pages[b]
    q = torch.randn((B, L, Hq, 128), generator=g, device="cuda").bfloat16()
    n_tok = np.array(lengths, np.int32)
    for call in range(2):
        out = torch.zeros((B, L, Hq, 128), dtype=torch.bfloat16, device="cuda")
        mass = torch.zeros((L * Hkv, NP * ps), device="cuda")
        st = md.lib().md_attend_mass_noalloc(pool.data_ptr(), bt.data_ptr(), n_tok.ctypes.data, q.data_ptr(),
                                             out.data_ptr(), mass.data_ptr(), B, L, Hq, Hkv, ps, P, NP,
                                             torch.cuda.current_stream().cuda_stream)
        assert st == md.MD_OK
        torch.cuda.synchronize()
        for b in range(B):
            n, pg = lengths[b], bt[b, :pages[b]].long()
            kv = pool[:, pg].double().transpose(1, 2)                  # [L][Hkv][pages][2][ps][128]
            k, v = (kv[:, :, :, i].reshape(L, Hkv, -1, 128)[:, :, :n] for i in (0, 1))
            p = torch.softmax(torch.einsum("lhgd,lhnd->lhgn", q[b].double().view(L, Hkv, G, 128), k) / 128 ** 0.5, -1)
            o = torch.einsum("lhgn,lhnd->lhgd", p, v).reshape(L, Hq, 128)
            assert float((out[b].double() - o).abs().max()) <= TOL_O_ABS, (call, b)
            want = p.sum(2).reshape(L * Hkv, n)
            slots = (pg[:, None] * ps + torch.arange(ps, device="cuda")).flatten()[:n]
            rel = ((mass[:, slots].double() - want).abs() / (want + TOL_FLOOR)).max()
            assert float(rel) <= TOL_REL, (call, b, float(rel))


@pytest.mark.parametrize("L,Hq,Hkv,ps,lengths", [
    (1, 16, 2, 16, [1]),
    (1, 12, 2, 32, [1703, 33]),
    (2, 16, 2, 16, [430 - 3 * i for i in range(32)]),
    *NOALLOC_PERSISTENT,
])
@pytest.mark.parametrize("stale", [0x7FFF, 0x7F80])          # a NaN and an infinity
def test_noalloc_ignores_what_lies_past_the_cached_tokens(L, Hq, Hkv, ps, lengths, stale):
    """Slots past a sequence's cached tokens may hold anything: NaN or infinite
    bits there give the same output and masses, bit for bit, as zeros."""
    B, P = len(lengths), max(lengths) // ps + 1
    pages = [(n + ps - 1) // ps for n in lengths]
    first = np.concatenate([[0], np.cumsum(pages)])
    g = torch.Generator(device="cuda").manual_seed(47)
    pool = torch.randn((L, int(first[-1]), Hkv, 2, ps, 128), generator=g, device="cuda").bfloat16().view(torch.int16)
    bt = torch.zeros((B, P), dtype=torch.int32)
    for b in range(B):
        bt[b, :pages[b]] = torch.arange(int(first[b]), int(first[b + 1]))
    bt = bt.cuda()
    q = torch.randn((B, L, Hq, 128), generator=g, device="cuda").bfloat16()
    n_tok = np.array(lengths, np.int32)
    got = []
    for bits in (0, stale):
        for b in range(B):
            if lengths[b] % ps:
                pool[:, int(first[b + 1]) - 1, :, :, lengths[b] % ps:] = bits
        out = torch.zeros((B, L, Hq, 128), dtype=torch.int16, device="cuda")
        mass = torch.zeros((L * Hkv, int(first[-1]) * ps), device="cuda")
        st = md.lib().md_attend_mass_noalloc(pool.data_ptr(), bt.data_ptr(), n_tok.ctypes.data, q.data_ptr(),
                                             out.data_ptr(), mass.data_ptr(), B, L, Hq, Hkv, ps, P, int(first[-1]),
                                             torch.cuda.current_stream().cuda_stream)
        assert st == md.MD_OK
        torch.cuda.synchronize()
        got.append((out, mass))
    assert torch.isfinite(got[1][0].view(torch.bfloat16).float()).all()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


def test_noalloc_rejects_work_beyond_its_fixed_scratch():
    """Too many (sequence, layer, KV head) items for the fixed array: a clear
    capacity error before anything is launched."""
    dummy = torch.zeros(64, dtype=torch.int32, device="cuda")
    n_tok = np.full(256, 4096, np.int32)
    p = dummy.data_ptr()
    st = md.lib().md_attend_mass_noalloc(p, p, n_tok.ctypes.data, p, p, p, 256, 36, 16, 2, 16, 4096, 64, None)
    assert st == md.MD_ERR_CAPACITY
    # the 3B geometry's full trace, 32 x 1,700 tokens: two chunks per item
    # would need about 37 MiB of scores and partials
    n_tok2 = np.full(32, 1700, np.int32)
    st = md.lib().md_attend_mass_noalloc(p, p, n_tok2.ctypes.data, p, p, p, 32, 36, 16, 2, 16, 107, 64, None)
    assert st == md.MD_ERR_CAPACITY
    st = md.lib().md_attend_mass_noalloc(p, p, n_tok.ctypes.data, p, p, p, 1, 2, 16, 2, 24, 4096, 64, None)
    assert st == md.MD_ERR_INVALID_ARG
    torch.cuda.synchronize()
