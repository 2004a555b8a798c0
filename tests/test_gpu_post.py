"""Device reductions after propagation: spectrum (Eqs. 15, 16) and group charges,
against the oracle's own propagation followed by the oracle's formulas."""
import numpy as np
import pytest

import oracle as O
from oracle import spectrum as OS
from paper_2308_09782_gb300 import inputs
from tests._gpu_util import oracle_ground, system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2308_09782_gb300 import vgtb
    vgtb.load()


def test_spectrum_of_a_kick_matches_oracle():
    from paper_2308_09782_gb300 import vgtb
    sysd, _, _ = system("si8_pulse")
    ctx, gs = oracle_ground("si8_pulse")
    n, a0 = 1500, 0.001
    A = inputs.kick_field(n, a0)
    ref_J = O.propagate(sysd, A, n, gs["D"], ctx=ctx)["J"]
    e0 = -a0 / O.C_LIGHT
    w = np.linspace(0.02, 1.0, 60)
    s_ref = OS.conductivity(ref_J, sysd["dt"], e0, w, 200.0)
    e_ref = OS.dielectric(s_ref, w)
    with vgtb.Context(sysd, init=vgtb.INIT_USER) as c:
        for k, D in enumerate(gs["D"]):
            c.set_density(0, k, D)
        c.set_field(0, A)
        c.propagate(n)
        s, e = c.spectrum(0, e0, w, tau0=200.0)
        s2, _ = c.spectrum(0, e0, w, n0=100, n1=900)
    assert np.abs(s - s_ref).max() <= 1e-8 * np.abs(s_ref).max()
    assert np.abs(e - e_ref).max() <= 1e-8 * np.abs(e_ref).max()
    t = np.arange(801) * sysd["dt"]
    assert np.abs(s2 - OS.conductivity(ref_J[100:901], sysd["dt"], e0, w, 200.0)).max() <= 1e-8 * np.abs(s2).max()
    assert np.abs(s[:, 0]).max() > 10 * np.abs(s[:, 1]).max()   # response along the kick
    del t


def test_group_charges_match_oracle_series():
    from paper_2308_09782_gb300 import vgtb
    sysd, A, _ = system("si64_pulse")
    ctx, gs = oracle_ground("si64_pulse")
    n = 300
    ref_q = O.propagate(sysd, A, n, gs["D"], ctx=ctx)["q"]
    # groups: coordination-like classes from a 5.0 bohr bond cutoff, plus "no group" atoms
    pos, lat = sysd["pos"], sysd["lattice"]
    d = pos[:, None, :] - pos[None, :, :]
    d -= np.round(d / lat[0, 0]) * lat[0, 0]
    coord = ((np.sqrt((d ** 2).sum(-1)) < 5.0).sum(1) - 1)
    group = np.where(coord >= 4, 1, 0).astype(np.int32)
    group[::7] = -1
    with vgtb.Context(sysd, init=vgtb.INIT_USER, obs_stride=3) as c:
        for k, D in enumerate(gs["D"]):
            c.set_density(0, k, D)
        c.set_field(0, A)
        c.propagate(n)
        dq = c.group_charges(0, group, 2)
    lv = np.arange(0, n + 1, 3)
    ref = np.stack([-(ref_q[lv][:, group == g] - ref_q[0, group == g]).sum(1) for g in range(2)], 1)
    assert dq.shape == ref.shape
    assert np.abs(dq - ref).max() <= 1e-10
    assert np.abs(ref).max() > 1e-6


def test_laser_sweep_coordination_charge_transfer_matches_oracle():
    """The laser experiment of Sec. 3.3 in small: three photon energies as three
    trajectories of one context (FP64), charge transfer per coordination class
    (2.85 A bond cut-off) against the oracle's charges of each single run."""
    from paper_2308_09782_gb300 import inputs, vgtb
    sysd = inputs.diamond_si(2, 0.3, seed=64, kgrid="gamma")
    ctx = O.setup(sysd)
    gs = O.ground_state(sysd, ctx=ctx)
    fields, _ = inputs.laser_sweep(sysd["dt"])
    n = 250
    cn = inputs.coordination_numbers(sysd)
    classes = sorted(set(cn.tolist()))
    assert len(classes) >= 2                          # the displacements break some bonds
    group = np.array([classes.index(c) for c in cn], np.int32)
    with vgtb.Context([sysd], traj_sys=[0, 0, 0], init=vgtb.INIT_USER) as c:
        c.set_density(0, 0, gs["D"][0])
        for tr, f in enumerate(fields):
            c.set_field(tr, f[:n + 1])
        c.propagate(n)
        got = [c.group_charges(tr, group, len(classes)) for tr in range(3)]
    moved = []
    for tr, f in enumerate(fields):
        q = O.propagate(sysd, f[:n + 1], n, gs["D"], ctx=ctx)["q"]
        ref = np.stack([-(q[:, group == g] - q[0, group == g]).sum(1) for g in range(len(classes))], 1)
        assert np.abs(got[tr] - ref).max() <= 1e-10
        moved.append(np.abs(ref).max())
    assert min(moved) > 1e-7                          # every pulse moved charge


def test_spectrum_takes_the_phases_without_rounding():
    """Every level's weight is e^{i w t} e^{-t/tau0} at the exact product w n dt.  Against the same sum over the
    device's own J with phases reduced in rational arithmetic: a sine or cosine is off by at most 2 ulp and
    an exp by 1 in either factor (12 x 2^-53), their product and those with J and the trapezoid weight round
    6 times, and 5 + 5 + 8 additions follow; here the reduced phase, cosine, exp and products make at most
    12: below 48 x 2^-53 of the sum of |terms|, 64 allowed.  (Phases rounded as w t are off by up to
    1e6 x 2^-53 at the highest frequency.)"""
    from fractions import Fraction
    from paper_2308_09782_gb300 import vgtb
    sysd, _, _ = system("si8_pulse")
    _, gs = oracle_ground("si8_pulse")
    n, a0, tau0 = 1200, 0.001, 200.0
    w = [0.05, 0.4, 373.0, 1207.0, 4001.0]
    with vgtb.Context(sysd, init=vgtb.INIT_USER) as c:
        for k, D in enumerate(gs["D"]):
            c.set_density(0, k, D)
        c.set_field(0, inputs.kick_field(n, a0))
        c.propagate(n)
        J, _, _ = c.observables(0)
        s, _ = c.spectrum(0, 1.0, np.array(w), tau0=tau0)
    turn = Fraction("6.283185307179586476925286766559005768394338798750211641949889")
    f = np.full(n + 1, sysd["dt"])
    f[[0, -1]] *= 0.5
    term = (f * np.exp(-np.arange(n + 1) * sysd["dt"] / tau0))[:, None] * J
    size = 64 * 2.0 ** -53 * np.abs(term).sum(0)
    for i, wi in enumerate(w):
        x = np.array([float(Fraction(wi) * Fraction(float(sysd["dt"])) * m % turn) for m in range(n + 1)])[:, None]
        assert np.all(np.abs(s[i].real - (np.cos(x) * term).astype(np.longdouble).sum(0)) <= size), wi
        assert np.all(np.abs(s[i].imag - (np.sin(x) * term).astype(np.longdouble).sum(0)) <= size), wi


def test_a_large_read_out_gives_its_buffer_back():
    """Charges of 2001 levels by 8192 groups are 131 MB on the device: as much is free after the call as before
    (an allocation's granularity of 2 MB aside), and a small call still answers."""
    import torch
    from paper_2308_09782_gb300 import vgtb
    sysd, _, _ = system("si8_pulse")
    _, gs = oracle_ground("si8_pulse")
    n = 2000
    with vgtb.Context(sysd, init=vgtb.INIT_USER) as c:
        for k, D in enumerate(gs["D"]):
            c.set_density(0, k, D)
        c.set_field(0, inputs.kick_field(n, 0.01))
        c.propagate(n)
        small = c.group_charges(0, np.arange(8, dtype=np.int32) % 2, 2)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        big = c.group_charges(0, np.arange(8, dtype=np.int32) % 2, 8192)
        assert torch.cuda.mem_get_info()[0] >= free - (2 << 20)
        assert np.array_equal(big[:, :2], small) and not big[:, 2:].any()
        assert np.array_equal(c.group_charges(0, np.arange(8, dtype=np.int32) % 2, 2), small)
