"""The FP64 path in residues on inputs that are not all of one size or one sign.

Reference: the DMMA kernel, which tc_energy_dev_noalloc always runs.  Its W elements carry 2^-51 to 2^-50, and an
energy is a sum over at least v^3 / 6 points of them.
"""
import numpy as np
import pytest

import paper_2512_01055_gb300 as tc
from tests.test_gpu_fp64_tensor import _energy, _noalloc, _random

pytestmark = pytest.mark.gpu


def test_long_sums_of_one_sign():
    """Operand rows that are constant along K at the longest K (1024): the residue sums reach 2^24, their bound."""
    import torch
    o, v = 2, 504
    d = _random(o, v, 404)
    g = torch.Generator(device="cuda").manual_seed(405)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    d["ovvv"] = (n(o, v) * 0.06)[:, :, None, None].expand(o, v, v, v).contiguous()
    h = (n(v) * 0.01)[:, None].expand(v, v)
    d["t2"][1, 0] = h
    d["t2"][0, 1] = h.T
    d["t2"][1, 1] = 0.01234
    r, e = _energy(o, v, d)
    assert r.prep_seconds > 0.0 and r.wterm_seconds < r.kernel_seconds          # residues, not the DMMA kernel
    e_ref, ref = _noalloc(o, v, d)
    scale = np.abs(ref).max()
    print(f"max |de| / max |e| = {np.abs(e - ref).max() / scale:.2e}")
    assert np.abs(e - ref).max() <= 1e-12 * scale
    assert abs(r.e_t - e_ref) <= 1e-12 * np.abs(ref).sum()


@pytest.mark.parametrize("what", ["t2", "ovvv and ovoo"])
def test_norms_whose_squares_underflow(what):
    """Operands at 2^-540: their squares are zero in FP64, their products with the other operands are not."""
    o, v = 4, 21
    d = _random(o, v, 93)
    for n in what.split(" and "):
        d[n] *= 2.0 ** -540
    r, e = _energy(o, v, d)
    e_ref, ref = _noalloc(o, v, d)
    assert np.abs(ref).max() > 0.0
    assert np.all(np.abs(e - ref) <= 1e-11 * np.abs(ref))
    assert abs(r.e_t - e_ref) <= 1e-12 * np.abs(ref).sum()


def _scale(d, what, k):
    """d with the named operands of one occupied or one virtual orbital (or a block of pairs) times 2^-k."""
    import torch
    o, v = d["t1"].shape
    d = {n: x.clone() for n, x in d.items()}
    f, p, x = 2.0 ** -k, 2, 5
    ints = what.startswith("ints")
    if what == "pairs":                             # weakly coupled orbitals: triplets of three are weak, others are not
        keep = torch.eye(o, dtype=torch.bool, device="cuda")[:, :, None, None]
        d["t2"] = torch.where(keep, d["t2"], d["t2"] * f)
        d["ovoo"] *= f
        return d
    if what in ("ovvv_occ", "ints_occ"):
        d["ovvv"][p] *= f
    if what in ("ovvv_vir", "ints_vir"):
        for a in range(1, 4):
            d["ovvv"].select(a, x).mul_(f)
    if what in ("ovoo_occ", "ints_occ"):
        for a in (0, 2, 3):
            d["ovoo"].select(a, p).mul_(f)
    if what in ("ovoo_vir", "ints_vir"):
        d["ovoo"][:, x] *= f
    if ints:
        axes = (0, 2) if what == "ints_occ" else (1, 3)
        for a in axes:
            d["ovov"].select(a, p if what == "ints_occ" else x).mul_(f)
    if what == "t2_occ":
        for a in (0, 1):
            d["t2"].select(a, p).mul_(f)
    if what == "t2_vir":
        for a in (2, 3):
            d["t2"].select(a, x).mul_(f)
    return d


WHAT = ["ovvv_occ", "ovvv_vir", "ovoo_occ", "ovoo_vir", "t2_occ", "t2_vir", "ints_occ", "ints_vir"]


@pytest.mark.parametrize("what", WHAT)
@pytest.mark.parametrize("k", [8, 16, 24, 32, 40])
def test_operands_of_one_orbital_smaller_than_the_others(what, k):
    o, v = 5, 24
    d = _scale(_random(o, v, 611), what, k)
    r, e = _energy(o, v, d)
    assert r.prep_seconds > 0.0 and r.wterm_seconds < r.kernel_seconds
    e_ref, ref = _noalloc(o, v, d)
    scale = np.abs(ref).max()
    print(f"{what} 2^-{k}: max |de| / max |e| = {np.abs(e - ref).max() / scale:.2e}, dE/E = {abs(r.e_t / e_ref - 1):.2e}")
    assert np.abs(e - ref).max() <= 1e-12 * scale
    assert abs(r.e_t - e_ref) <= 1e-12 * np.abs(ref).sum()


# A triplet's W is right to 2^-49 of its own size (the weakest the residues are used for), the reference's to 2^-50;
# e_ijk may cancel between its W and V parts: three orders of magnitude over that.
@pytest.mark.parametrize("what", WHAT + ["pairs"])
@pytest.mark.parametrize("k", [6, 12, 20, 30])
def test_every_triplet_keeps_its_own_digits(what, k):
    o, v = 6, 21
    d = _scale(_random(o, v, 612), what, k)
    r, e = _energy(o, v, d)
    assert r.prep_seconds > 0.0
    e_ref, ref = _noalloc(o, v, d)
    nz = ref != 0.0
    worst = np.abs(e[nz] / ref[nz] - 1).max()
    print(f"{what} 2^-{k}: worst relative error of a triplet {worst:.2e}")
    assert worst <= 1e-11
    assert abs(r.e_t - e_ref) <= 1e-12 * np.abs(ref).sum()


def test_served_job_with_weak_triplets():
    """A job some of whose triplets are formed again gives the same bits alone and served, beside one with none."""
    jobs = [(6, 21, _scale(_random(6, 21, 612), "pairs", 20)), (5, 24, _random(5, 24, 613))]
    alone = [_energy(*j)[0] for j in jobs]
    strong = _energy(6, 21, _random(6, 21, 612))[0]
    assert alone[0].launches > strong.launches                       # some triplets were weak
    ctx = tc.tc_init(0, max_inflight=4)
    try:
        for _ in range(2):
            tickets = [tc.tc_submit(ctx, o, v, d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"], d["ovov"],
                                    prec=tc.TC_FP64, device_inputs=True) for o, v, d in jobs]
            for t, a in zip(tickets, alone):
                code, r = tc.tc_wait(ctx, t, 60000)
                assert code == tc.TC_OK
                assert r.e_t == a.e_t and r.e_t5 == a.e_t5
        st = tc.tc_serve_stats_get(ctx)
        assert st.completed == 4 and st.failed == 0 and st.reserved_bytes == 0 and st.inflight == 0
    finally:
        tc.tc_finalize(ctx)


def test_inputs_beyond_the_grid_do_not_run_the_residue_products():
    """The call notices them after its preparation: what it does besides the DMMA kernel is a small part of a call."""
    o, v = 8, 104
    d = _random(o, v, 95)
    good = min((_energy(o, v, d)[0] for _ in range(3)), key=lambda r: r.seconds)
    d["ovvv"][2, 3, 4, 5] = float("inf")
    bad = min((_energy(o, v, d)[0] for _ in range(3)), key=lambda r: r.seconds - r.kernel_seconds)
    assert bad.prep_seconds == 0.0 and bad.kernel_seconds > 5 * good.kernel_seconds
    print(f"good {good.seconds:.4f} s, of it residue kernels {good.kernel_seconds:.4f} s; "
          f"beside the DMMA kernel {bad.seconds - bad.kernel_seconds:.4f} s")
    assert bad.seconds - bad.kernel_seconds < 0.5 * good.kernel_seconds


# o = 2, v = 9: the smallest shape of the residues; v = 8, o = 1 and K beyond 1024 take the DMMA kernel
@pytest.mark.parametrize("o,v,residues", [(2, 9, True), (2, 8, False), (1, 12, False), (3, 9, True), (9, 10, True),
                                          (2, 504, True), (2, 505, False)])
def test_which_kernel_runs(o, v, residues):
    d = _random(o, v, 900 + v)
    r, e = _energy(o, v, d)
    assert (r.prep_seconds > 0.0) == residues and (r.wterm_seconds < r.kernel_seconds) == residues
    e_ref, ref = _noalloc(o, v, d)
    assert np.abs(e - ref).max() <= 1e-12 * np.abs(ref).max()
    assert abs(r.e_t - e_ref) <= 1e-12 * np.abs(ref).sum()


@pytest.mark.parametrize("spread", [3, 6, 9])
def test_factors_per_orbital_keep_the_residues(spread):
    """Every orbital's integrals and amplitudes times its own factor between 2^-spread and 1: the exponents take the
    factors out, and no triplet needs the DMMA kernel (which would show in the number of launches)."""
    import torch
    o, v = 6, 40
    d = _random(o, v, 78)
    launches = _energy(o, v, d)[0].launches
    g = torch.Generator(device="cuda").manual_seed(6)
    fo, fv = (torch.exp2(-spread * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)) for n in (o, v))
    d["ovvv"] *= fo[:, None, None, None] * fv[None, :, None, None] * fv[None, None, :, None] * fv
    d["ovoo"] *= fo[:, None, None, None] * fv[None, :, None, None] * fo[None, None, :, None] * fo
    d["t2"] *= fo[:, None, None, None] * fo[None, :, None, None] * fv[None, None, :, None] * fv
    r, e = _energy(o, v, d)
    e_ref, ref = _noalloc(o, v, d)
    nz = ref != 0.0
    print(f"spread 2^-{spread}: {r.launches - launches} launches more, worst relative error of a triplet "
          f"{np.abs(e[nz] / ref[nz] - 1).max():.2e}")
    assert r.launches == launches
    assert np.all(np.abs(e - ref) <= 1e-11 * np.abs(ref))
    assert abs(r.e_t - e_ref) <= 1e-12 * np.abs(ref).sum()
