"""CPU models of the weight-gradient kernels' staging as it is now (csrc/conv_wgrad.cuh,
csrc/conv_wgrad_ring.cuh): row segments of any multiple of 16 pixels up to 160, chosen by padding
and hand-overs, and channel groups an odd number of 16-byte rows apart.  The tap-row model of
test_wgrad_models.py runs with such plans (exact integer sums through staging, descriptor reads and
scatter, every address inside the allocation); of the ring, the parts that differ from its model
there: the gradient slot and the order in which the activation's copies are issued."""
import numpy as np
import pytest

import test_wgrad_models as models
from test_wgrad_models import BUDGET, MAX_STAGES, MAX_UNITS, PRODUCERS, TAPROW_SHAPES, UM, _read_plain, _tiles

MAX_SEG, STAGE_COST, PAD_G, PAD_X = 160, 32, 1, 3
RING_MIN_STAGES, RING_MAX_G_UNITS, TAP_MIN_STAGES = 3, 4, 4


def _segments(W):
    """Segments from the longest down, and the cost by which the first cheapest that fits is taken."""
    for seg in range((W + 15) // 16 * 16 if W < MAX_SEG else MAX_SEG, 15, -16):
        yield seg, (W + seg - 1) // seg * (seg + STAGE_COST)


def taprow_plan(B, H, W, Cin, Cout, sms=152):
    ntg, ng = _tiles(Cin)
    ntx, nx = _tiles(Cout)
    mtg, mtx = (Cout + UM - 1) // UM, (Cin + UM - 1) // UM
    xa = mtx * ntx * nx < mtg * ntg * ng
    a = dict(xa=xa, m_tiles=mtx if xa else mtg, n_tiles=ntx if xa else ntg, N=nx if xa else ng)
    a["ngA"], a["ngB"] = min(16, ((Cin if xa else Cout) + 7) // 8), a["N"] // 8
    a["ncombo"] = 3 * a["m_tiles"] * a["n_tiles"]
    ngx, ngg = (a["ngA"], a["ngB"]) if xa else (a["ngB"], a["ngA"])
    best = None
    for seg, cost in _segments(W):
        if best is not None and cost >= best:
            continue
        nk = seg // 16
        lenA, lenB = (seg + PAD_X, seg + PAD_G) if xa else (seg + PAD_G, seg + PAD_X)
        As, Bs = a["ngA"] * lenA * 16, a["ngB"] * lenB * 16
        if (16 * (nk - 1) + (0 if xa else 2)) * 16 + (a["ngB"] - 1) * lenB * 16 + 256 > Bs:
            continue
        if ngx * (seg + 2) > MAX_UNITS * PRODUCERS or ngg * seg > MAX_UNITS * PRODUCERS:
            continue
        for S in range(MAX_STAGES, TAP_MIN_STAGES - 1, -1):
            total = max(S * (As + Bs), (S - 1) * As + (16 * (nk - 1) + (2 if xa else 0)) * 16 + 15 * lenA * 16 + 256)
            if total <= BUDGET:
                best = cost
                a.update(seg=seg, nk=nk, lenA=lenA, lenB=lenB, a_slot=As, b_slot=Bs, b_ring=S * As, stages=S,
                         smem=total)
                break
    a["nseg"] = (W + a["seg"] - 1) // a["seg"]
    a["total"] = B * H * a["nseg"]
    per = (a["total"] * a["ncombo"] + sms - 1) // sms
    a["lb"] = min(256, max(8, per // 3))
    a["f_total"] = (a["total"] + a["lb"] - 1) // a["lb"] * a["ncombo"] * a["lb"]
    a["f_per_cta"] = (a["f_total"] + sms - 1) // sms
    a["grid"] = (a["f_total"] + a["f_per_cta"] - 1) // a["f_per_cta"]
    return a


@pytest.mark.parametrize("shape", TAPROW_SHAPES + [(1, 2, 132, 64, 64), (1, 1, 264, 96, 32), (1, 2, 66, 128, 128)])
def test_taprow_model_with_odd_group_pitches_gives_the_direct_sums(shape, monkeypatch):
    monkeypatch.setattr(models, "taprow_plan", taprow_plan)
    a, got, want = models.run_taprow(*shape)
    assert a["smem"] <= BUDGET and a["lenA"] % 2 and a["lenB"] % 2
    assert np.array_equal(got, want)


@pytest.mark.parametrize("N", [16, 32, 48, 128])
@pytest.mark.parametrize("seg", [16, 32, 112, 144, 160])
def test_ring_gradient_slot(seg, N):
    """Channel group i, pixel p at (i (seg + 1) + p) 16 bytes: each K step's descriptor reads the
    16 pixels it names of every channel, inside the slot."""
    if N // 8 * seg > RING_MAX_G_UNITS * PRODUCERS:
        pytest.skip("not planned: more copies than a producer's table holds")
    pitch = seg + PAD_G
    smem = np.full(N // 8 * pitch * 8, np.nan)
    g = np.arange(seg * N, dtype=float).reshape(seg, N)
    for i in range(N // 8):
        for p in range(seg):
            smem[(i * pitch + p) * 8:(i * pitch + p) * 8 + 8] = g[p, 8 * i:8 * i + 8]
    for kk in range(seg // 16):
        B = _read_plain(smem, 16 * kk * 16, pitch * 16, N)
        assert np.array_equal(B, g[16 * kk:16 * kk + 16].T)


@pytest.mark.parametrize("ncc", [2, 4])
def test_ring_activation_copies_cover_a_row_without_bank_conflicts(ncc):
    """The pixels of a group of eight are staged in bit-reversed order: every (tap, pixel, group) once,
    and the eight threads that write at a time hit eight different 16-byte chunks of the 128-byte
    rows' banks (tap by tap, away from a wrap of the group index)."""
    seg, n_atoms = 32, (3 * ncc * 8 + 63) // 64
    seen = set()
    for u0 in range(0, 3 * ncc * seg, 8):
        chunks = []
        for u in range(u0, u0 + 8):
            q, grp = divmod(u, ncc)
            tx = q // seg
            pl = q - tx * seg
            p = (pl & ~5) | (pl & 1) << 2 | (pl >> 2 & 1)
            seen.add((tx, p, grp))
            mg, r8 = tx * ncc + grp, p & 7
            dst = ((p >> 3) * n_atoms + (mg >> 3)) * 1024 + r8 * 128 + ((mg & 7) ^ r8) * 16
            chunks.append(dst // 16 % 8)
        assert len(set(chunks)) == 8, (u0, chunks)
    assert seen == {(t, p, c) for t in range(3) for p in range(seg) for c in range(ncc)}
