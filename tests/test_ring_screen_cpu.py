"""The ring form of the FP32 screen (csrc/screen.cuh: ring_vertex, ring_values,
ring_bound), which the screened pass uses: compiled for the host and run on
the adversarial triangle families of the screen's other test.  With one bound
for both sides of the move, from the larger radius and the smaller edge sum,
and the step's number packed into the low bits, 2 sqrt(3) times every packed
value must lie within ring_bound of alpha in binary128 and in the FP64 tree."""
import os
import re
import tempfile

import pytest

import test_screen_bounds as tsb


def _harness():
    """The families and reference alphas of the other test, with its check of
    the two sides replaced by the ring form's."""
    a = tsb.HARNESS.index("    const float sk = slot == 1")
    b = tsb.HARNESS.index("    /* the difference screen: the sign it claims")
    e = tsb.HARNESS.index("static P rot(double r, double th)")
    check = r"""
    /* P -> Q in the stored direction: A, B for slots 0 and 2, B, A for slot 1 */
    float h[4] = {0, 0, 0, 0}, hA[4], hB[4];
    head_tail(bits(p.x), h[0], h[1]); head_tail(bits(p.y), h[2], h[3]);
    head_tail(bits(A.x), hA[0], hA[1]); head_tail(bits(A.y), hA[2], hA[3]);
    head_tail(bits(B.x), hB[0], hB[1]); head_tail(bits(B.y), hB[2], hB[3]);
    const RingVertex vA = ring_vertex(hA[0], hA[1], hA[2], hA[3], h[0], h[1], h[2], h[3], Cx, Cy);
    const RingVertex vB = ring_vertex(hB[0], hB[1], hB[2], hB[3], h[0], h[1], h[2], h[3], Cx, Cy);
    float v[2], s[2];
    if (slot == 1) ring_values(vB, vA, v[0], v[1], s[0], s[1]);
    else ring_values(vA, vB, v[0], v[1], s[0], s[1]);
    const float smin = fminf(s[0], s[1]), g = side_g(fmaxf(rn, rC), smin);
    if (!ring_ok(smin, g)) { ++n_bound_fail; return; }
    const float bnd = ring_bound(g);
    for (int side = 0; side < 2; ++side) {
        const uint32_t step = (uint32_t)(nxt() & 15u);
        const float packed = with_step(v[side], step);
        if (step_of(packed) != step) ++n_bad;
        const float a = kTwoSqrt3f * packed;
        const P node = side ? c : p;
        const P t0 = stored(slot, 0, node, A, B), t1 = stored(slot, 1, node, A, B), t2 = stored(slot, 2, node, A, B);
        const double a64 = alpha64(t0, t1, t2);
        const qreal aq = alphaq(t0, t1, t2);
        double eq = (double)((qreal)a - aq);
        eq = eq < 0 ? -eq : eq;
        const double e64 = fabs((double)a - a64);
        ++n_checked;
        if (eq / bnd > worst_q) worst_q = eq / bnd;
        if (e64 / bnd > worst_64) worst_64 = e64 / bnd;
        if (!(eq <= (double)bnd) || !(e64 <= (double)bnd)) {
            if (n_bad < 10) printf("BAD fam %d side %d slot %d a %.9g fp64 %.17g bound %.3g g %.3g\n", fam, side, slot,
                                   (double)a, a64, (double)bnd, (double)g);
            ++n_bad;
        }
    }
}

"""
    return tsb.HARNESS[:a] + check + tsb.HARNESS[e:]


def _run(header_dir, per, shift):
    with tempfile.TemporaryDirectory() as d:
        old, tsb.HARNESS = tsb.HARNESS, _harness()
        try:
            exe = tsb._build(d, header_dir)
        finally:
            tsb.HARNESS = old
        return tsb._run(exe, per, shift)


@pytest.mark.parametrize("shift", [-2, 0, 2])
def test_ring_bound(shift):
    rc, out = _run(tsb.CSRC, 450_000, shift)
    assert rc == 0, out
    m = re.search(r"checked (\d+) .* worst_q ([\d.]+) worst_64 ([\d.]+) bad 0", out)
    assert m and int(m.group(1)) >= 400_000, out
    assert float(m.group(2)) < 1.0 and float(m.group(3)) < 1.0, out


def test_a_weaker_ring_bound_is_caught():
    hdr = open(os.path.join(tsb.CSRC, "screen.cuh")).read()
    weak = hdr.replace("return side_bound(1.05f, g) + kPackEps;", "return 0.03f * side_bound(1.05f, g);")
    assert weak != hdr
    with tempfile.TemporaryDirectory() as d:
        with open(os.path.join(d, "screen.cuh"), "w") as f:
            f.write(weak)
        rc, out = _run(d, 100_000, 0)
        assert rc != 0 and "BAD" in out, out
