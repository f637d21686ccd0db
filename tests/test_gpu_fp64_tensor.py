"""The FP64 path on the tensor cores (residue products) at the edges of its tiles.

References: the CPU oracle, and for shapes whose oracle would be slow the
DMMA kernel, which tc_energy_dev_noalloc always runs.

Tolerance.  W is rounded once to a grid about 2^-53 of its size and E_T sums
W^2-like terms; the oracle and the DMMA kernel carry about 2^-51 per W element
and a few 2^-53 per sum.  All of it averages out over v^3 points, so 1e-12 of
the largest triplet contribution leaves three orders of magnitude over what
any of them commits, and three under the path's 1e-9 bound.
"""
import numpy as np
import pytest

import oracle
import synth
import paper_2512_01055_gb300 as tc
from tests import gpu_util

pytestmark = pytest.mark.gpu
TOL = 1e-12


def _noalloc(o, v, d):
    import torch
    e_t = torch.zeros(1, dtype=torch.float64, device="cuda")
    e_ijk = torch.zeros((o,) * 3, dtype=torch.float64, device="cuda")
    tc.tc_energy_dev_noalloc(o, v, d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"], d["ovov"], e_t, e_ijk=e_ijk)
    torch.cuda.synchronize()
    return float(e_t.item()), e_ijk.cpu().numpy()


def _energy(o, v, d):
    import torch
    e_ijk = torch.zeros((o,) * 3, dtype=torch.float64, device="cuda")
    r = tc.tc_energy_dev(gpu_util.context(), o, v, d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"], d["ovov"],
                         prec=tc.TC_FP64, e_ijk=e_ijk)
    return r, e_ijk.cpu().numpy()


def _random(o, v, seed):
    """Device inputs of the synthetic jobs' sizes without a factor (ovvv symmetric in its last pair)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    u = lambda k, a, b: torch.sort(a + (b - a) * torch.rand(k, generator=g, device="cuda", dtype=torch.float64)).values
    ovvv = n(o, v, v, v) * 0.06
    ovvv = ((ovvv + ovvv.transpose(2, 3)) * 0.5).contiguous()
    ovoo = n(o, v, o, o) * 0.06
    ovov = n(o * v, o * v) * 0.06
    t2 = n(o * v, o * v) * 0.01
    return dict(eps=torch.cat([u(o, -1.5, -0.3), u(v, 0.1, 3.0)]), t1=n(o, v) * 0.005,
                t2=((t2 + t2.T) * 0.5).reshape(o, v, o, v).permute(0, 2, 1, 3).contiguous(), ovvv=ovvv,
                ovoo=((ovoo + ovoo.transpose(2, 3)) * 0.5).contiguous(),
                ovov=((ovov + ovov.T) * 0.5).reshape(o, v, o, v).contiguous())


# v = 8 the smallest; 9, 17: N padding; 15, 16: one N group; 23, 24: K halves;
# o = 2: only triplets with equal indices; o = 9: two K halves over occupied
@pytest.mark.parametrize("o,v,seed", [(2, 8, 1), (3, 9, 2), (4, 15, 3), (3, 16, 4), (5, 17, 5), (2, 24, 6), (9, 23, 7),
                                      (8, 33, 8)])
def test_small_shapes_match_oracle(o, v, seed):
    job = synth.make_job(o, v, seed)
    r, e_ijk = gpu_util.energy_dev(job, want_trip=True)
    ref = {t: oracle.triplet_energy(job, *t) for t in oracle.triplet_list(o)}
    scale = max(abs(x) for x in ref.values())
    for t, x in ref.items():
        assert abs(e_ijk[t] - x) <= TOL * scale, (t, e_ijk[t], x)
    e4, e5 = oracle.energy_parts_eq1(job)
    assert abs(r.e_t5 - e5) <= TOL * (abs(e4) + abs(e5))


# 160, 161: the drain's sums in registers alone, then some in tensor memory;
# 208, 209: the widest N chunk, then two; 504: the largest K (1024); 505: beyond it
@pytest.mark.parametrize("o,v", [(3, 100), (4, 160), (3, 161), (2, 208), (3, 209), (2, 300), (2, 504), (2, 505)])
def test_wide_shapes_match_the_dmma_kernel(o, v):
    d = _random(o, v, 1000 + v)
    r, e = _energy(o, v, d)
    e_ref, ref = _noalloc(o, v, d)
    scale = np.abs(ref).max()
    print(f"o={o} v={v} max |de| / max |e| = {np.abs(e - ref).max() / scale:.2e}")
    assert np.abs(e - ref).max() <= TOL * scale
    assert abs(r.e_t - e_ref) <= TOL * np.abs(ref).sum()


def test_triplet_subset_makes_only_the_images_it_reads():
    job = synth.make_job(7, 40, 71)
    d = gpu_util.to_device(job)
    _, e_ijk = gpu_util.energy_dev(job, want_trip=True, dev=d)
    for trip in ([(6, 6, 2)], [(5, 1, 1), (5, 1, 1)], [(6, 4, 3), (2, 1, 0), (3, 3, 1)]):
        e, _ = tc.tc_triplets_dev(gpu_util.context(), 7, 40, d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"],
                                  d["ovov"], trip)
        assert all(e[m] == e_ijk[t] for m, t in enumerate(trip))


@pytest.mark.parametrize("spread", [0, 4, 8])
def test_orbitals_of_uneven_size(spread):
    """Every orbital's integrals and amplitudes scaled by its own factor between 2^-spread and 1."""
    import torch
    o, v = 5, 48
    d = _random(o, v, 77)
    g = torch.Generator(device="cuda").manual_seed(5)
    fo, fv = (torch.exp2(-spread * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)) for n in (o, v))
    d["ovvv"] *= fo[:, None, None, None] * fv[None, :, None, None] * fv[None, None, :, None] * fv[None, None, None, :]
    d["ovoo"] *= fo[:, None, None, None] * fv[None, :, None, None] * fo[None, None, :, None] * fo[None, None, None, :]
    d["t2"] *= fo[:, None, None, None] * fo[None, :, None, None] * fv[None, None, :, None] * fv[None, None, None, :]
    r, e = _energy(o, v, d)
    e_ref, ref = _noalloc(o, v, d)
    nz = ref != 0.0
    print(f"spread 2^-{spread}: worst relative error of a triplet {np.abs(e[nz] / ref[nz] - 1).max():.2e}")
    assert np.all(np.abs(e - ref) <= 1e-11 * np.abs(ref))
    assert abs(r.e_t - e_ref) <= TOL * np.abs(ref).sum()


@pytest.mark.parametrize("what", ["huge", "tiny", "nan", "inf"])
def test_inputs_beyond_the_integer_grid_take_the_dmma_kernel(what):
    o, v = 4, 21
    d = _random(o, v, 91)
    if what == "huge":
        d["ovvv"] *= 2.0 ** 130
        d["ovoo"] *= 2.0 ** 130
    elif what == "tiny":
        d["t2"] *= 2.0 ** -130
    else:
        d["ovvv"][2, 3, 4, 5] = float(what)
    r, e = _energy(o, v, d)
    e_ref, ref = _noalloc(o, v, d)
    assert np.array_equal(np.isfinite(e), np.isfinite(ref))
    ok = np.isfinite(ref)
    assert np.all(np.abs(e[ok] - ref[ok]) <= TOL * np.abs(ref[ok]).max())
    assert np.isfinite(r.e_t) == np.isfinite(e_ref)


def test_zero_operands():
    """All-zero ovvv or ovoo or t2: one of the two products of W vanishes, or W itself."""
    o, v = 4, 19
    for zero in ("ovvv", "ovoo", "t2"):
        d = _random(o, v, 93)
        d[zero].zero_()
        r, e = _energy(o, v, d)
        e_ref, ref = _noalloc(o, v, d)
        assert np.all(np.abs(e - ref) <= TOL * max(np.abs(ref).max(), 1e-300)), zero


def test_batched_jobs_of_different_widths_give_the_bits_of_each_alone():
    """Several FP64 jobs in one launch, their N chunks (48 to 208 columns) meeting in one pipeline."""
    shapes = [(4, 40), (3, 100), (2, 200), (5, 33), (3, 170), (4, 64), (2, 209)]
    devs = [_random(o, v, 300 + n) for n, (o, v) in enumerate(shapes)]
    alone = [_energy(o, v, d)[0] for (o, v), d in zip(shapes, devs)]
    ctx = tc.tc_init(0, max_inflight=8)
    try:
        assert tc.tc_inject_fault(ctx, tc.TC_FAULT_STALL, 400) == tc.TC_OK      # all are ready before the first launch
        tickets = [tc.tc_submit(ctx, o, v, d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"], d["ovov"],
                                prec=tc.TC_FP64, device_inputs=True) for (o, v), d in zip(shapes, devs)]
        for t, a in zip(tickets, alone):
            code, r = tc.tc_wait(ctx, t, 60000)
            assert code == tc.TC_OK
            assert r.e_t == a.e_t and r.e_t5 == a.e_t5
        st = tc.tc_serve_stats_get(ctx)
        assert st.batched_jobs > st.iterations
    finally:
        tc.tc_finalize(ctx)


# (4, 48) holds about 51 MB of images and W: no room for them; room, given back after the call; kept
@pytest.mark.parametrize("budget_mb,kept", [(16, False), (128, False), (1024, True)])
def test_images_within_the_budget_and_given_back(budget_mb, kept):
    import torch
    o, v = 4, 48
    d = _random(o, v, 48)
    e_ref, ref = _noalloc(o, v, d)
    e_ijk = torch.zeros((o,) * 3, dtype=torch.float64, device="cuda")
    ctx = tc.tc_init(0, hbm_budget_bytes=budget_mb << 20)
    try:
        args = (ctx, o, v, d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"], d["ovov"])
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(2):
            r = tc.tc_energy_dev(*args, prec=tc.TC_FP64, e_ijk=e_ijk)
            assert np.abs(e_ijk.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()
            assert abs(r.e_t - e_ref) <= TOL * np.abs(ref).sum()
            assert (free - torch.cuda.mem_get_info()[0] > 32 << 20) == kept
    finally:
        tc.tc_finalize(ctx)
