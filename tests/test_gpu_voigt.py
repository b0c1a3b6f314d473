"""The Voigt function as the kernels evaluate it (mpsa_voigt, through the C ABI) against the
FP64 oracle H = Re w(v + ia), per tier, on a (v, a) grid that spans every tier boundary."""
import numpy as np
import pytest

from oracle.voigt import H

pytestmark = pytest.mark.gpu

# relative-error bounds per tier (FP32 evaluation; derived from the tier truncation errors
# plus a few FP32 roundings: far <= 1e-6 + rounding, mid and core ~ 3e-6)
FP32_RTOL = 5e-6
FP64_RTOL = 1e-11


def grid():
    a = np.geomspace(1e-5, 30.0, 61)
    v = np.r_[0.0, np.geomspace(1e-3, 1e7, 700)]
    # points hugging the tier boundaries |z|^2 = 36 and 1600 and the rational-form switch
    extra_v = []
    for aa in a:
        for z2 in (36.0, 1600.0, 1000.0 * np.sqrt(2 + 2 * aa * aa)):
            for f in (1 - 1e-6, 1 + 1e-6):
                if z2 * f > aa * aa:
                    extra_v.append((np.sqrt(z2 * f - aa * aa), aa))
    V, A = np.meshgrid(v, a, indexing="ij")
    V, A = V.ravel(), A.ravel()
    ev = np.array(extra_v)
    return np.r_[V, ev[:, 0]], np.r_[A, ev[:, 1]]


def device_H(ctx, v, a, prec):
    import torch
    tv = torch.from_numpy(v).cuda()
    ta = torch.from_numpy(a).cuda()
    out = torch.empty_like(tv)
    ctx.voigt(tv, ta, out, precision=prec)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def test_fp32_tiers_against_oracle():
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    v, a = grid()
    vf, af = v.astype(np.float32).astype(np.float64), a.astype(np.float32).astype(np.float64)
    g = device_H(ctx, vf, af, binding.PREC_FP32_COMPENSATED)
    o = H(vf, af)
    rel = np.abs(g / o - 1)
    z2 = vf * vf + af * af
    for name, m in (("core", z2 < 36), ("mid", (z2 >= 36) & (z2 < 1600)), ("far", z2 >= 1600)):
        assert m.any()
        assert rel[m].max() <= FP32_RTOL, (name, rel[m].max(), vf[m][np.argmax(rel[m])], af[m][np.argmax(rel[m])])
    ctx.close()


def test_fp64_tiers_against_oracle():
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    v, a = grid()
    g = device_H(ctx, v, a, binding.PREC_FP64)
    o = H(v, a)
    rel = np.abs(g / o - 1)
    assert rel.max() <= FP64_RTOL, (rel.max(), v[np.argmax(rel)], a[np.argmax(rel)])
    ctx.close()


def test_weakly_damped_and_series_forms_against_oracle():
    # the profile's form for a <= 0.03 inside |z| = 10 (both of its branches, down to the damping of
    # low-pressure lines) and the series outside it, hugging their boundaries.  Where e^{-V} makes up
    # H, rounding V = v^2 costs V 2^-24, 2e-6 at V = 34 (a = 1e-16; beyond it the wing takes over)
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    e = 1e-6
    a = np.r_[np.geomspace(1e-16, 0.03, 60), 3e-4 * (1 - e), 3e-4 * (1 + e), 0.03 * (1 - e), 0.03 * (1 + e), 0.3, 3.0, 30.0]
    v = np.r_[0.0, np.linspace(1e-3, 10.2, 2500), np.geomspace(10.0, 1e4, 200)]
    V, A = (x.ravel() for x in np.meshgrid(v, a, indexing="ij"))
    edge = [(np.sqrt(100.0 * f - x * x), x) for x in a if x < 9.9 for f in (1 - e, 1 + e)]
    V, A = np.r_[V, [x for x, _ in edge]], np.r_[A, [y for _, y in edge]]
    vf, af = V.astype(np.float32).astype(np.float64), A.astype(np.float32).astype(np.float64)
    rel = np.abs(device_H(ctx, vf, af, binding.PREC_FP32_COMPENSATED) / H(vf, af) - 1)
    assert rel.max() <= FP32_RTOL, (rel.max(), vf[np.argmax(rel)], af[np.argmax(rel)])
    ctx.close()


@pytest.mark.parametrize("form", ["POINT", "PAIR", "NODE"])
def test_profile_forms_against_oracle(form):
    # the forms of the profile kernel beside those of the cut windows (the two tests above): points on their own,
    # packed pairs, wing nodes, over every damping and hugging |z|^2 = 64 and 100 (the series' edges, a^2 <= 2 and
    # above), a = 3e-4, 0.03 and sqrt 2, and the rational form's switch
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    e = 1e-6
    a = np.r_[np.geomspace(1e-16, 1e3, 115), [x * (1 + s * e) for x in (3e-4, 0.03, np.sqrt(2.0)) for s in (-1, 1)]]
    v = np.r_[0.0, np.linspace(1e-3, 10.2, 1200), np.geomspace(10.0, 1e7, 300)]
    V, A = (x.ravel() for x in np.meshgrid(v, a, indexing="ij"))
    edge = [(np.sqrt(z * f - x * x), x) for x in a for z in (64.0, 100.0, 1e3 * np.sqrt(2 + 2 * x * x))
            for f in (1 - e, 1 + e) if z * f > x * x]
    V, A = np.r_[V, [x for x, _ in edge]], np.r_[A, [y for _, y in edge]]
    vf, af = V.astype(np.float32).astype(np.float64), A.astype(np.float32).astype(np.float64)
    rel = np.abs(device_H(ctx, vf, af, getattr(binding, "VOIGT_" + form)) / H(vf, af) - 1)
    assert rel.max() <= FP32_RTOL, (rel.max(), vf[np.argmax(rel)], af[np.argmax(rel)])
    ctx.close()


def test_line_centre_against_oracle_and_tiers():
    # H(0, a) of the line terms: within the tiers' error of the oracle, and within rounding of the core tier, which
    # forms the two poles of a pair apart (terms of one sign, some 30 roundings: 2e-6)
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    a = np.r_[np.geomspace(1e-16, 1e4, 4000), [x * (1 + s * 1e-6) for x in (2.0, 6.0) for s in (-1, 1)]]
    a = a.astype(np.float32).astype(np.float64)
    g, t = (device_H(ctx, v, a, p) for v, p in ((np.full_like(a, 7.0), binding.VOIGT_CENTRE), (np.zeros_like(a), 0)))
    assert np.abs(g / H(np.zeros_like(a), a) - 1).max() <= FP32_RTOL
    assert np.abs(g / t - 1).max() <= 2e-6
    ctx.close()


def test_cut_window_tiers_of_weak_damping():
    # the tiers that decide the cut windows, down to the damping of low-pressure lines (test_fp32_tiers above starts
    # at a = 1e-5): where e^{-v^2} makes up H its argument's rounding costs v^2 2^-24, 2e-6 at v^2 = 36
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    a = np.geomspace(1e-16, 1e-5, 40)
    v = np.r_[0.0, np.linspace(1e-3, 10.2, 2500), np.geomspace(10.0, 1e4, 200)]
    V, A = (x.ravel() for x in np.meshgrid(v, a, indexing="ij"))
    vf, af = V.astype(np.float32).astype(np.float64), A.astype(np.float32).astype(np.float64)
    rel = np.abs(device_H(ctx, vf, af, binding.PREC_FP32_COMPENSATED) / H(vf, af) - 1)
    assert rel.max() <= FP32_RTOL, (rel.max(), vf[np.argmax(rel)], af[np.argmax(rel)])
    ctx.close()


def test_weak_damping_has_no_step():
    # a <= 3e-4 inside |z| = 10 (the terms in a^3 and a^4 left out, 8e-8 in all) and just above it: the error of
    # ex2.approx (2^-22), of the reciprocal and of some FP32 roundings of the quotient leave less than 1e-6
    from paper_2105_13611_gb300 import binding
    ctx = binding.Context(0)
    a = np.r_[np.geomspace(1e-8, 3e-4, 40), 3.001e-4, 4e-4]
    V, A = (x.ravel() for x in np.meshgrid(np.linspace(0.0, 9.99, 5000), a, indexing="ij"))
    vf, af = V.astype(np.float32).astype(np.float64), A.astype(np.float32).astype(np.float64)
    rel = np.abs(device_H(ctx, vf, af, binding.VOIGT_POINT) / H(vf, af) - 1)
    assert rel.max() <= 1e-6, (rel.max(), vf[np.argmax(rel)], af[np.argmax(rel)])
    ctx.close()
