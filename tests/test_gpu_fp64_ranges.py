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
