"""The kernels' internal paths at the sizes where they can go wrong: chunks of
candidates, near ties of equal codes, the lookup table's element lists, signed
NVFP4 codes, the symmetric codes' clamp sets and candidates of equal sums,
weights and saliencies at the ends of fp32's range, and launches around the
number of CTAs or warps that the device holds."""
import json

import numpy as np
import pytest
import torch

from paper_2608_13966_gb300 import api, quasar, workloads as wl
from tests import checker
from tests import gpu_harness as H
from tests.test_parity_gpu import CLIP8, NARROW8, _assert, _edge_inputs, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clip", [wl.CLIP_16[:9], wl.CLIP_PAPER, wl.CLIP_16,
                                  tuple(1.0 - 0.02 * i for i in range(17)),
                                  tuple(0.3 + 0.02 * i for i in range(32)),
                                  (0.9, 0.3, 0.6, 1.0, 0.5, 0.8, 0.4, 0.7, 0.95, 0.35)],
                         ids=["9", "paper", "16", "17", "32_up", "10_unordered"])
@pytest.mark.parametrize("bits,G", [(2, 64), (3, 128), (4, 32), (2, 256)])
def test_int_chunks_of_candidates(oracle, clip, bits, G):
    """More than 8 candidates: a partial last chunk, factors in decreasing,
    increasing and no order, degenerate groups, a ragged last unit."""
    w, g, v = _inputs(7, 21 * G, seed=4000 + bits)
    w[0] = 0.25                                            # zero range
    v[1] = 0.0; g[1] = 0.0                                 # all saliency zero
    w[3, ::2] = 0.0                                        # many exact zeros
    w[4, 5] = 3.0                                          # one outlier
    w[5] = torch.linspace(-1, 1, 21 * G, device="cuda")    # codes on grid boundaries
    w[6] += 5.0                                            # far from zero
    _assert(*H.run_int(oracle, w, g, v, bits=bits, group_size=G, clip=list(clip),
                       r_dtype=torch.float32))


@pytest.mark.parametrize("bits,K", [(2, 8), (2, 16), (1, 8), (3, 8)])
def test_int_ties_between_runs_of_equal_codes(oracle, bits, K):
    """Groups of two tight clusters and one weight between them, of a saliency
    from far below to near the others': the candidates fall into runs of equal
    codes, and the runs' errors differ by little beside the explained part (the
    case where the kept candidate is picked among twins)."""
    gen = torch.Generator(device="cuda").manual_seed(7 + bits)
    n, G = 4096, 128
    u = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    w = torch.where(u(n, G) < 0.5, -1.0, 1.0) * (1.0 + 1e-3 * (u(n, G) - 0.5))
    w[:, 17] = u(n) * 1.8 - 0.9
    v = 1e-6 * (0.5 + u(n, G))
    v[:, 17] = 1e-6 * 10.0 ** (-9.0 * u(n))
    _assert(*H.run_int(oracle, w, None, v, bits=bits, group_size=G, clip=list(wl.CLIP_16[:K]),
                       r_dtype=torch.float32))


def _lut_case(oracle, w, v, clip):
    w_h, v_h = H._host(w), H._host(v)
    o = api.recon_lut_batch([(w, None, v)], clip=clip, codes=True)[0]
    torch.cuda.synchronize()
    w2, h2 = w_h.reshape(w.shape), v_h.reshape(w.shape)
    O = oracle.recon_lut(w2, h2, clip)
    gpu = {"r": H._host(o["r"]), "book": o["book"].cpu().numpy(),
           "codes": o["codes"].cpu().numpy(), "idx": o["cand_idx"].cpu().numpy()}
    rep = checker.check_lut(oracle, w2, h2, clip, O, gpu)
    assert rep["ok"], json.dumps(rep)


@pytest.mark.parametrize("K", [1, 8, 9, 32])
@pytest.mark.parametrize("kind", ["all", "one_side", "counts"])
def test_lut_element_lists(oracle, kind, K):
    """Blocks whose lists of elements that reach level 1 hold all 512 weights
    (both signs, or 511 of one), or from 2 to 65 of them."""
    clip = [round(1.0 - 0.7 * i / max(K - 1, 1), 4) for i in range(K)]
    gen = torch.Generator(device="cuda").manual_seed(11)
    n = 64
    u = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    if kind == "all":
        x = torch.where(u(n, 512) < 0.5, -1.0, 1.0) * (0.5 + 0.5 * u(n, 512))
    elif kind == "one_side":
        x = 0.6 + 0.4 * u(n, 512)
        x[:, 100] = -1.0
    else:  # block i: i + 2 weights far out, the rest close to the centre
        x = 0.02 * (u(n, 512) - 0.5)
        x[:, 0], x[:, 511] = -1.0, 1.0
        for i in range(n):
            k = 1 + torch.randperm(510, generator=gen, device="cuda")[:i]
            x[i, k] = torch.where(u(i) < 0.3, -1.0, 1.0) * (0.3 + 0.7 * u(i))
    w = (0.05 * x).reshape(n, 8, 64).permute(1, 0, 2).reshape(8, n * 64).contiguous()
    v = torch.exp(-14.0 + 2.0 * torch.randn(w.shape, generator=gen, device="cuda"))
    _lut_case(oracle, w, v, clip)


@pytest.mark.parametrize("K", [1, 3, 7, 9, 15])
def test_nvfp4_signs_zeros_and_candidate_counts(oracle, K):
    """Negative weights that round to a code of magnitude 0, zeros of either
    sign and zero blocks: code 0 and r = +0, in every output format."""
    clip = [round(1.0 - 0.6 * i / max(K - 1, 1), 4) for i in range(K)]
    w, g, v = _inputs(24, 512, seed=4200 + K)
    w[0, ::2] = -1e-9
    w[1] = -0.0
    w[2, ::3] = 0.0
    _assert(*H.run_nvfp4(oracle, w.clone(), g, v.clone(), clip=clip))
    one = api.recon_nvfp4_batch([(w, g, v.clone())], clip=clip, codes=True, r_dtype=torch.float32)[0]
    two = api.recon_nvfp4_batch([(w, g, v.clone())], clip=clip, codes=True, packed_codes=True)[0]
    torch.cuda.synchronize()
    codes = one["codes"].cpu().numpy().ravel()
    assert np.array_equal(oracle.unpack_nvfp4_codes(two["codes"].cpu().numpy()), codes)
    assert not (codes == 8).any()
    r = one["r"].cpu().numpy()
    assert not np.signbit(r[r == 0]).any()


@pytest.mark.parametrize("bits,clip", [(2, CLIP8), (3, CLIP8), (4, CLIP8), (4, NARROW8),
                                       (3, wl.CLIP_16), (3, wl.CLIP_PAPER), (8, CLIP8)],
                         ids=["sets8", "sets4", "sets332", "sets8_int4", "k16", "paper", "sets1"])
@pytest.mark.parametrize("G", [32, 64, 128, 256])
def test_sym_clamp_sets_equal_per_candidate_clamp(bits, clip, G):
    """|w| capped once per set of candidates gives bit for bit the outputs of
    the cap of every candidate on its own (checked against the oracle in the
    parity tests), on ragged shapes with degenerate groups."""
    outs = {}
    try:
        for hoist in (True, False):
            quasar.quasar_debug_set_hoist(hoist)
            items = [_edge_inputs(r, c, seed=4300 + i) for i, (r, c) in
                     enumerate([(37, 3 * G), (8, 2 * G), (1, G)])]
            outs[hoist] = api.recon_int_batch(items, bits=bits, group_size=G, clip=list(clip),
                                              codes=True, symmetric=True)
            torch.cuda.synchronize()
    finally:
        quasar.quasar_debug_set_hoist(True)
    for a, b in zip(outs[True], outs[False]):
        for key in ("r", "a", "b", "codes", "cand_idx"):
            assert torch.equal(a[key], b[key]), key


@pytest.mark.parametrize("units", [1, 7, 151, 153, 303, 305, 2431, 2433, 3647, 3649])
@pytest.mark.parametrize("kind", ["int", "sym", "nvfp4", "lut"])
def test_launches_around_the_number_of_ctas(kind, units):
    """As many units of work as the 152 SMs, twice as many, or as warps (16 an SM,
    NVFP4 24), more or less one: the outputs equal those of the same weights
    passed as two tensors."""
    rows, cols = {"int": (8 * units, 32), "sym": (8 * units, 32), "nvfp4": (units, 512),
                  "lut": (8 * units, 64)}[kind]
    w, g, v = _inputs(rows, cols, seed=4400 + units)
    cut = rows // 8 // 2 * 8 if kind != "nvfp4" else rows // 2

    def run(items):
        if kind == "nvfp4":
            amax = w.abs().max().reshape(1)
            return api.recon_nvfp4_batch([(*it, amax) for it in items], clip=CLIP8, codes=True)
        if kind == "lut":
            return api.recon_lut_batch(items, clip=CLIP8, codes=True)
        return api.recon_int_batch(items, bits=3, group_size=32, clip=CLIP8, codes=True,
                                   symmetric=kind == "sym")

    whole = run([(w, g, v.clone())])[0]
    parts = run([(w[:cut], g[:cut], v[:cut].clone()), (w[cut:], g[cut:], v[cut:].clone())])
    torch.cuda.synchronize()
    for key in whole:
        if key != "tensor_scale":
            assert torch.equal(whole[key], torch.cat([p[key] for p in parts])), key


@pytest.mark.parametrize("G,g_dtype,adam,symmetric", [
    (32, torch.bfloat16, False, False), (128, torch.float32, False, False),
    (256, torch.bfloat16, False, False), (256, None, False, False), (64, torch.bfloat16, True, False),
    (128, torch.bfloat16, True, False), (256, torch.bfloat16, True, False), (256, torch.float32, True, False),
    (32, None, False, True), (128, torch.bfloat16, False, True), (256, torch.float32, False, True)])
def test_tiles_shared_by_the_warps_of_a_cta(G, g_dtype, adam, symmetric):
    """Every slot of a CTA's ring is filled several times, for each number of
    slots and warps: the outputs equal those of calls small enough that each
    slot is filled once at most."""
    rows, piece = 8 * (152 * 40 + 5), 8 * 152 * 4          # one group a row, 8 a tile
    w, g, v = _inputs(rows, G, seed=4500 + G)
    m = 1e-4 * torch.randn(rows, G, device="cuda", generator=torch.Generator("cuda").manual_seed(G))
    g = None if g_dtype is None else g.to(g_dtype)

    def run(lo, hi):
        cut = lambda x: None if x is None else x[lo:hi].clone()
        wc, gc, mc, vc = cut(w), cut(g), cut(m), cut(v)
        if adam:
            out = api.adamw_recon_int_batch([(wc, gc, mc, vc)], bits=3, group_size=G, clip=CLIP8, lr=1e-5,
                                             step=3)[0]
        else:
            out = api.recon_int_batch([(wc, gc, vc)], bits=3, group_size=G, clip=CLIP8, codes=True,
                                      symmetric=symmetric)[0]
        return dict(out, w=wc, m=mc, v=vc)

    whole = run(0, rows)
    parts = [run(lo, min(lo + piece, rows)) for lo in range(0, rows, piece)]
    torch.cuda.synchronize()
    for key in whole:
        if whole[key] is not None:
            assert torch.equal(whole[key], torch.cat([p[key] for p in parts])), key


@pytest.mark.parametrize("g_dtype,adam", [(torch.bfloat16, False), (torch.float32, False), (None, False),
                                          (torch.bfloat16, True), (torch.float32, True)])
def test_nvfp4_warps_that_begin_with_the_next_stage(g_dtype, adam):
    """A batch in several stages (some warps of a launch take the absmax or the
    AdamW step of the next stage's tensors first, then reconstruct): the outputs
    equal those of one call a tensor.  A small last tensor, a ragged row."""
    shapes = [(4099, 2048), (4096, 2064), (8200, 1024), (3, 16)]
    items = []
    for i, (r, c) in enumerate(shapes):
        w, g, v = _inputs(r, c, seed=4600 + i)
        m = 1e-4 * torch.randn(r, c, device="cuda", generator=torch.Generator("cuda").manual_seed(i))
        items.append((w, None if g_dtype is None else g.to(g_dtype), m, v))

    def run(items):
        items = [tuple(None if x is None else x.clone() for x in it) for it in items]
        if adam:
            out = api.adamw_recon_nvfp4_batch(items, clip=CLIP8, codes=True, lr=1e-5, step=3)
        else:
            out = api.recon_nvfp4_batch([(w, g, v) for w, g, _, v in items], clip=CLIP8, codes=True)
        return [dict(o, w=it[0], m=it[2], v=it[3]) for o, it in zip(out, items)]

    whole = run(items)
    single = [run([it])[0] for it in items]
    torch.cuda.synchronize()
    for a, b in zip(whole, single):
        for key in a:
            if a[key] is not None:
                assert torch.equal(a[key], b[key]), key


def _small_weights(rows, G, seed):
    """Groups (one a row) of multiples of 2^-12, zeros among them, which a power
    of two scales without rounding down to 2^-137."""
    w, _, v = _inputs(rows, G, seed=seed)
    w = torch.round(w * 4096.0) / 4096.0
    w[0], w[1, ::2] = 0.0, 0.0
    w[2] = (torch.arange(G, device="cuda") * 5 % 7 - 3) / 4096.0
    w[3] += 0.125                                          # one sign, a small range
    return w, v


@pytest.mark.parametrize("e", [-22, -100, -122, -135])
@pytest.mark.parametrize("bits,G,clip", [(2, 64, CLIP8), (4, 128, CLIP8), (8, 32, wl.CLIP_16),
                                         (4, 256, (1.0, 0.25)), (3, 128, (1.0, 0.5, 1e-30, 1e-37))],
                         ids=["int2", "int4", "int8_k16", "int4_two", "tiny_factors"])
@pytest.mark.parametrize("kind", ["sym", "int", "adamw"])
def test_weights_scaled_by_a_power_of_two(oracle, kind, bits, G, clip, e):
    """Groups of weights down to the smallest denormals keep the factor and the
    codes that the same weights have at their usual size, and a fit and an r
    smaller by the power of two (both code layouts; an AdamW step of rate 0)."""
    w, v = _small_weights(40, G, seed=4700 + bits)
    s = 2.0 ** e

    def run(w, packed):
        kw = dict(bits=bits, group_size=G, clip=list(clip), codes=True, packed_codes=packed,
                  r_dtype=torch.float32)
        v1, z = v.clone(), torch.zeros_like(w)
        if kind == "adamw":
            w1 = w.clone()
            o = api.adamw_recon_int_batch([(w1, z, z.clone(), v1)], lr=0.0, step=1, **kw)[0]
            assert torch.equal(w1, w)
        else:
            o = api.recon_int_batch([(w, None, v1)], symmetric=kind == "sym", **kw)[0]
        torch.cuda.synchronize()
        return dict(o, v=v1)

    ref, small, packed = run(w, False), run(w * s, False), run(w * s, True)
    for key in ("codes", "cand_idx"):
        assert torch.equal(small[key], ref[key]), key
    assert np.array_equal(oracle.unpack_int_codes(packed["codes"].cpu().numpy(), bits, w.numel()),
                          small["codes"].cpu().numpy().ravel())
    for key in ("r", "a", "b"):
        want, got = ref[key].double() * s, small[key].double()
        # both sides within 1e-7 + 1e-5 |x| at a size about 1 (ref's own: 0.1),
        # and the spacing of the denormals, of which r sums up to 256
        lim = 2e-5 * want.abs() + s * 2e-7 + 256 * 2.0 ** -149
        assert bool(((got - want).abs() <= lim).all()), key  # (a NaN fails)
        assert torch.equal(packed[key], small[key]), key
    w_h, h = H._host(w * s), H._host(small["v"])
    O = (oracle.recon_sym if kind == "sym" else oracle.recon_int)(w_h, h, G, bits, list(clip))
    same = (O["m_round"] >= checker.MARGIN) & (O["m_tie"] >= checker.MARGIN)
    assert np.array_equal(small["cand_idx"].cpu().numpy()[same], O["idx"][same])


@pytest.mark.parametrize("bits,K", [(2, 8), (2, 16), (3, 8), (4, 16), (8, 8)])
@pytest.mark.parametrize("descending", [True, False])
def test_sym_ties_between_runs_of_equal_codes(oracle, bits, K, descending):
    """Groups of two tight clusters and one weight between them, of a saliency
    so far below the others' that its codes do not move the fp32 sums: factors
    of equal sums have different codes and errors."""
    gen = torch.Generator(device="cuda").manual_seed(17 + bits)
    n, G = 2048, 128
    u = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    w = torch.where(u(n, G) < 0.5, -1.0, 1.0)
    w[n // 2:] *= 1.0 + 1e-4 * (u(n - n // 2, G) - 0.5)
    w[:, 17] = u(n) * 1.8 - 0.9
    v = 1e-6 * (0.5 + u(n, G))
    v[:, 17] = 1e-6 * 10.0 ** (-10.0 * u(n))
    clip = list(wl.CLIP_16[:K]) if descending else list(wl.CLIP_16[:K])[::-1]
    if descending and K == 16:
        clip = clip[1::2] + clip[::2]                      # in no order
    w_h, h = H._host(w), H._host(v)
    o = api.recon_int_batch([(w, None, v)], bits=bits, group_size=G, clip=clip, codes=True, symmetric=True,
                            r_dtype=torch.float32)[0]
    torch.cuda.synchronize()
    O = oracle.recon_sym(w_h, h, G, bits, clip)
    gpu = {"r": H._host(o["r"]), "a": o["a"].cpu().numpy(), "b": o["b"].cpu().numpy(),
           "codes": o["codes"].cpu().numpy().ravel(), "idx": o["cand_idx"].cpu().numpy()}
    rep = checker.check_sym(oracle, w_h, h, bits, clip, O, gpu, G, False)
    assert rep["ok"], json.dumps(rep)


@pytest.mark.parametrize("bits,G", [(3, 128), (8, 32)])
def test_sym_saliencies_scaled_by_a_power_of_two(bits, G):
    """Saliencies as large as their type holds give the outputs of the same ones
    at their usual size: a common scale of h changes nothing."""
    w, _, v = _inputs(40, G, seed=4800 + bits)
    v = v.clamp(max=0.5)
    outs = []
    for e in (0, 64, 126):
        outs.append(api.recon_int_batch([(w, None, v * 2.0 ** e)], bits=bits, group_size=G, clip=CLIP8,
                                        codes=True, symmetric=True)[0])
        torch.cuda.synchronize()
    for o in outs[1:]:
        for key in ("r", "a", "b", "codes", "cand_idx"):
            assert torch.equal(o[key], outs[0][key]), key


def test_nvfp4_first_factor_of_overflowing_moments(oracle):
    """Saliencies so large that the moments of the smaller factors, which come
    first, overflow (their codes are larger), and those of the last do not: a
    factor whose error is finite is kept, as the oracle keeps it."""
    clip = [0.3, 0.35, 1.0]
    w = torch.zeros(8, 16, device="cuda")
    v = torch.full((8, 16), 1e-6, device="cuda")
    w[:, 0] = 400.0                                        # code 6 for every factor
    w[:, 3], v[:, 3] = 132.0, 2e37                         # code 6 at 0.3 and 0.35, else 2
    rep, ema = H.run_nvfp4(oracle, w, None, v, clip=clip, r_dtype=torch.float32)
    _assert(rep, ema)
