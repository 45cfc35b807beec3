"""The ring form of the FP32 screen, and the difference screen after it, under
the condition that the pass itself puts on a node's local frame: by its furthest
neighbour alone, so that rings with one neighbour much nearer than 2^-20 of the
node's coordinates are screened too.  The same harness as the ring form's other test, with that condition, and
families in which one vertex of the triangle lies 2^-1 to 2^-45 of the other's
distance from the node (the move of the node's size, of the near neighbour's,
or onto it)."""
import os
import re
import tempfile

import pytest

import test_ring_screen_cpu as ring
import test_screen_bounds as tsb

NEAR = r"""
        if (k & 1) {
            const double da = hypot(A.x - p.x, A.y - p.y), near = da * ldexp(uni(0.5, 1.0), -(int)(nxt() % 45));
            B = add(p, rot(near, uni(0.0, 6.283185307179586)));
            switch (nxt() & 3) {
            case 0: c = add(p, rot(near * uni(0.0, 2.0), uni(0.0, 6.3))); break;
            case 1: c = add(B, rot(near * uni(0.0, 0.1), uni(0.0, 6.3))); break;
            case 2: c = add(p, rot(da * uni(0.0, 0.7), uni(0.0, 6.3))); break;
            default: break;  /* the family's own */
            }
            if (nxt() & 1) { const P t = A; A = B; B = t; }
        }
        check(fam, p, A, B, c, slot, rho);
"""


# settle_open's bound: each side's own radius, edge sum and quality, no step number
SIDES = r"""
    for (int side = 0; side < 2; ++side) {
        const float a1 = kTwoSqrt3f * v[side], g1 = side_g(side ? fmaxf(rn, rC) : rn, s[side]);
        if (!bound_ok(s[side], g1, fabsf(a1))) continue;
        const float b1 = side_bound(fabsf(a1), g1);
        const P node = side ? c : p;
        const P t0 = stored(slot, 0, node, A, B), t1 = stored(slot, 1, node, A, B), t2 = stored(slot, 2, node, A, B);
        double e1 = (double)((qreal)a1 - alphaq(t0, t1, t2));
        e1 = e1 < 0 ? -e1 : e1;
        if (!(e1 <= (double)b1) || !(fabs((double)a1 - alpha64(t0, t1, t2)) <= (double)b1)) {
            if (n_bad < 10) printf("BAD side fam %d side %d bound %.3g g %.3g\n", fam, side, (double)b1, (double)g1);
            ++n_bad;
        }
        ++n_sides;
        if (e1 / b1 > worst_side) worst_side = e1 / b1;
    }
    const float smin = fminf(s[0], s[1])"""


def _harness():
    b = tsb.HARNESS.index("    /* the difference screen: the sign it claims")
    e = tsb.HARNESS.index("static P rot(double r, double th)")
    h = ring._harness()
    end = "        }\n    }\n}\n\nstatic P rot(double r, double th)"  # of the ring form's check
    assert h.count(end) == 1
    h = h.replace(end, "        }\n    }\n    {\n" + tsb.HARNESS[b:e] + "}\n\nstatic P rot(double r, double th)")
    for old, new in (("!frame_ok(rmin, fmaxf(rn, rC), M)", "!frame_ok(rn, fmaxf(rn, rC), M)"),
                     ("        check(fam, p, A, B, c, slot, rho);\n", NEAR),
                     ("    const float smin = fminf(s[0], s[1])", SIDES),
                     ("static double worst_q = 0.0,", "static long n_sides = 0;\nstatic double worst_side = 0.0, worst_q = 0.0,"),
                     ('    printf("triangles %ld', '    printf("sides %ld worst_side %.4f\\n", n_sides, worst_side);\n    printf("triangles %ld')):
        assert h.count(old) == 1
        h = h.replace(old, new)
    return h


def _run(header_dir, per, shift):
    with tempfile.TemporaryDirectory() as d:
        old, tsb.HARNESS = tsb.HARNESS, _harness()
        try:
            exe = tsb._build(d, header_dir)
        finally:
            tsb.HARNESS = old
        return tsb._run(exe, per, shift)


def test_the_kernel_asks_the_same():
    text = open(os.path.join(tsb.CSRC, "pass_screened.cu")).read()
    assert "frame_ok(m.rn, rN, M)" in text and "const float rN = fmaxf(m.rn," in text
    assert "frame_ok(rn, rN, M) & bound_ok(smin, g, amax)" in text and "side_g(after ? rN : rn, smin)" in text


@pytest.mark.parametrize("shift", [-2, 0, 2])
def test_bound_and_difference_screen(shift):
    rc, out = _run(tsb.CSRC, 600_000, shift)
    assert rc == 0, out
    m = re.search(r"checked (\d+) frame_fail (\d+) .* diff_decided (\d+)/\d+ worst_q ([\d.]+) worst_64 ([\d.]+) bad 0", out)
    assert m and int(m.group(1)) >= 500_000 and int(m.group(3)) >= 50_000, out
    assert float(m.group(4)) < 1.0 and float(m.group(5)) < 1.0, out
    m = re.search(r"sides (\d+) worst_side ([\d.]+)", out)
    assert m and int(m.group(1)) >= 500_000 and float(m.group(2)) < 1.0, out


def test_a_weaker_frame_is_caught():
    # planted mistake: frames 2^12 times smaller than allowed, whose splits no
    # longer resolve the ring
    hdr = open(os.path.join(tsb.CSRC, "screen.cuh")).read()
    weak = hdr.replace("constexpr float kLocalRange = 1048576.0f;", "constexpr float kLocalRange = 1048576.0f * 65536.0f;")
    assert weak != hdr
    far = _harness().replace("h = M * ldexp(1.0, -20) * uni(1.0, 1.3);", "h = M * ldexp(1.0, -30) * uni(1.0, 1.3);")
    assert far != _harness()
    with tempfile.TemporaryDirectory() as d:
        with open(os.path.join(d, "screen.cuh"), "w") as f:
            f.write(weak)
        old, tsb.HARNESS = tsb.HARNESS, far
        try:
            exe = tsb._build(d, d)
        finally:
            tsb.HARNESS = old
        rc, out = tsb._run(exe, 100_000, 0)
        assert rc != 0 and "BAD" in out, out
