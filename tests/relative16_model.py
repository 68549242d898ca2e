"""Bit-level CPU model of the packed band kernel's relative frame (test infrastructure).

Restates, in plain Python integers, the arithmetic of ``lockstep16_loop`` in
``paper_2309_07270_gb300/csrc/xd_lockstep16.cuh`` for one group of lanes, with
the cells kept relative to each diagonal's X-drop threshold:
the substitution folded into one multiply-add, signed three-way maxima, the
prune by an unsigned add-and-minimum, the plain slot keys, the lift of
pruned slots and the window shifts.  Every add is checked: a half that
carries into the other one, or leaves the signed 16-bit range where the
kernel compares signed, raises Wrap.  Any change to the kernel's arithmetic
must be made here too.
"""
from packed16_model import Wrap, fits, mk, pack2, prmt, s16, uhalves, umk

DEAD = 0xC000
DEAD2 = 0xC000C000


def key_scale(slots):
    return max(slots, 16)


def slot_bits(slots):
    return {16: 4, 32: 5, 64: 6}[key_scale(slots)]


def relative_ok(match, mismatch, gap, x, slots):
    return (fits(match, mismatch, gap, x)
            and (x + 2 * match - 2 * gap + 1) * key_scale(slots) <= 0x8000
            and (slots < 64 or match - gap <= 64))


def subst_folds(match, mismatch, gap):
    mm, bonus = mismatch - 2 * gap, match - mismatch
    c = 2 * mm // bonus
    return c * bonus == 2 * mm and not c & 2 and c < 0x800


def lift_period(match, gap, slots):
    step = (match - gap) * key_scale(slots)
    return max(((1 << 14) // step - 2) // 2, 1)


def add(a, b):
    """A plain 32-bit add of two packed registers (no carry between halves);
    a live half (not negative) must stay below 2^15."""
    la, ha = uhalves(a)
    lb, hb = uhalves(b)
    for v, w in ((la, lb), (ha, hb)):
        if v < 0x8000 and v + w >= 0x8000:
            raise Wrap((v, w))
    return umk(la + lb, ha + hb)


def max_s(*v):
    lo = max(s16(x) for x in v)
    hi = max(s16(x >> 16) for x in v)
    return mk(lo, hi)


def addmin_u(a, b, c):
    la, ha = uhalves(a)
    lb, hb = uhalves(b)
    for v, w in ((la, lb), (ha, hb)):  # a pruned half must not wrap to a live one
        if v >= 0x8000 and s16(v) - (0x10000 - w) < -0x8000:
            raise Wrap((v, w))
    return umk(min((la + lb) & 0xFFFF, c & 0xFFFF), min((ha + hb) & 0xFFFF, c >> 16))


def flags(eqs, t, C2):
    """Register t's flag word and the bit of its low flag (rel_pos)."""
    if C2 == 2:
        e = (eqs[0] & 0xF) | (eqs[0] << 12 & 0xFFFFFFFF)
    elif C2 == 4:
        e = prmt(eqs[0], eqs[0], 0x2100)
    elif C2 == 8:
        e = eqs[0]
    else:
        h = t // 8
        e = prmt(eqs[h // 2], eqs[len(eqs) // 2 + h // 2], 0x7632 if h & 1 else 0x5410)
    G = 3 if C2 >= 16 else 2
    q = (t % 8) % G
    return e >> (2 * G * ((t % 8) // G)), q


def extend(a, b, match, mismatch, gap, x, lanes=2, regs=16, stats=None):
    """As packed16_model.extend, in the relative frame."""
    stats = {} if stats is None else stats
    for k in ("up", "down", "lift", "masked", "folded"):
        stats.setdefault(k, 0)
    C2, S = regs, 2 * regs
    KS, SB = key_scale(S), slot_bits(S)
    VS = SB if lanes == 1 else SB + 5
    W, m, n, ng = lanes * S, len(a), len(b), -gap
    NSH = max(min(S // 4, W // 8), 1)
    assert relative_ok(match, mismatch, gap, x, S)
    mm, bonus = mismatch + 2 * ng, match - mismatch
    folds = subst_folds(match, mismatch, gap)
    stats["folded"] += folds
    c = (2 * mm // bonus) * 0x10001 if folds else 0
    mi2 = 0 if folds else pack2(mm * KS)
    K = [bonus * KS >> (1 + 2 * q) for q in range(3)]
    period = lift_period(match, gap, S)

    def base_a(i):
        return int(a[i - 1]) if 1 <= i <= m else (i * 7 + 1) & 3

    def base_b(j):
        return int(b[j - 1]) if 1 <= j <= n else (j * 5 + 2) & 3

    E = [[DEAD2] * C2 for _ in range(lanes)]
    O = [[DEAD2] * C2 for _ in range(lanes)]
    for g in range(lanes):
        for t in range(C2):
            lo = x * KS if g * S + t == W // 2 else DEAD
            hi = x * KS if g * S + t + C2 == W // 2 else DEAD
            E[g][t] = umk(lo, hi)
    i0 = [-(W // 2) + g * S for g in range(lanes)]
    j0 = [(W // 2) - g * S for g in range(lanes)]
    st = dict(d=0, T=0, best=None, dA=ng, dB=ng)

    def margin():
        return min(m - (i0[0] + W - 1), n - j0[0])

    def diagonal(odd, masked):
        st["d"] += 1
        for g in range(lanes):
            if odd:
                i0[g] += 1
            else:
                j0[g] += 1
        if not masked and margin() < 0:
            raise AssertionError("unmasked diagonal leaves the rectangle")
        V, Uraw = (O, E) if odd else (E, O)
        dA, dB = pack2(st["dA"] * KS), pack2(st["dB"] * KS)
        nstep = (0x10000 - (dA + dB)) & 0xFFFFFFFF
        assert uhalves(nstep) == (0x10000 - (st["dA"] + st["dB"]) * KS,) * 2
        U = [[add(u, dA) for u in row] for row in Uraw]
        group = None
        newV = []
        for g in range(lanes):
            eqs = []
            for w0 in range(0, max(S, 16), 16):
                xx = 0
                for s in range(16):
                    xx |= ((base_a(i0[g] + w0 + s) ^ base_b(j0[g] - w0 - s)) & 3) << (2 * s)
                eqs.append(~(xx | (xx << 1)) & 0xFFFFFFFF)
                if masked:  # flags of the slots inside the rectangle only
                    lo, hi = j0[g] - n - w0, m - i0[g] - w0
                    keep = sum(3 << (2 * s) for s in range(16) if lo <= s <= hi)
                    eqs[-1] &= keep
            if odd:
                edge = U[g + 1][0] if g + 1 < lanes else DEAD2
            else:
                edge = U[g - 1][C2 - 1] if g > 0 else DEAD2
            row, lane = [], -0x8000
            for t in range(C2):
                if odd:
                    sh = U[g][t + 1] if t + 1 < C2 else prmt(U[g][0], edge, 0x5432)
                else:
                    sh = U[g][t - 1] if t > 0 else prmt(edge, U[g][C2 - 1], 0x5432)
                e, q = flags(eqs, t, C2)
                w = (e & (0x10001 << (1 + 2 * q))) | ((c << (2 * q)) & 0xFFFFFFFF)
                assert w * K[q] <= 0xFFFFFFFF
                cand = add(add(V[g][t], w * K[q]), mi2)
                r = max_s(cand, U[g][t], sh)
                v = addmin_u(r, nstep, DEAD2)
                row.append(v)
                idx = (S - 1 - t) | ((S - 1 - (t + C2)) << 16)
                key = add(r, idx)
                lane = max(lane, s16(key), s16(key >> 16))
            newV.append(row)
            mask = (1 << SB) - 1
            mkey = lane if lanes == 1 else 32 * lane - 31 * (lane & mask) + ((31 - g) << SB)
            assert mkey >> VS == lane >> SB
            group = mkey if group is None else max(group, mkey)
        for g in range(lanes):
            V[g][:] = newV[g]
        above = (group >> VS) - (st["dA"] + st["dB"])
        rise = max(above - x, 0)
        st["T"] += rise
        st["dA"], st["dB"] = st["dB"], ng + rise
        if rise:
            st["best"] = (group, i0[0], st["d"])
        return above

    def shift(up):
        for X in (E, O):
            if up:
                nx = [X[g + 1][0] if g + 1 < lanes else DEAD2 for g in range(lanes)]
                for g in range(lanes):
                    X[g] = X[g][1:] + [prmt(X[g][0], nx[g], 0x5432)]
            else:
                pv = [X[g - 1][C2 - 1] if g > 0 else DEAD2 for g in range(lanes)]
                for g in range(lanes):
                    X[g] = [prmt(pv[g], X[g][C2 - 1], 0x5432)] + X[g][:-1]
        for g in range(lanes):
            i0[g] += 1 if up else -1
            j0[g] -= 1 if up else -1

    def lo_live(v):
        return not v & 0x8000

    def hi_live(v):
        return not v >> 31

    budget, left, refill, prev_dead, top = margin(), period, 16, False, lanes - 1
    while True:
        masked = budget < 1
        stats["masked"] += masked
        dead_o = diagonal(True, masked) < 0
        dead_e = diagonal(False, masked) < 0
        fin = (dead_o and (prev_dead or dead_e)) or st["d"] >= m + n
        prev_dead = dead_e
        budget -= 1
        if fin:
            if st["best"] is None:
                return st["T"], 0, 0, False
            key, ibase, bd = st["best"]
            bi = ibase + S - 1 - (key & ((1 << SB) - 1))
            bi += 0 if lanes == 1 else (31 - ((key >> SB) & 31)) * S
            return st["T"], bi, bd - bi, False
        need_up = hi_live(E[top][C2 - 1]) or hi_live(O[top][C2 - 1])
        need_dn = lo_live(E[0][0])

        def free_bottom(k):
            return not any(lo_live(E[0][q]) for q in range(k + 1)) and \
                not any(lo_live(O[0][q]) for q in range(k))

        def free_top(k):
            return not any(hi_live(X[top][C2 - 1 - q]) for X in (E, O) for q in range(k + 1))
        if need_up or need_dn:
            free = free_bottom if need_up else free_top
            if not free(1):
                return st["T"], 0, 0, True
            by = NSH if free(NSH) else 1
            stats["up" if need_up else "down"] += by
            for _ in range(by):
                shift(need_up)
            budget = margin()
        refill -= 1
        if refill == 0:
            refill = 16
            if masked:  # end what lives outside the rectangle
                for g in range(lanes):
                    for X, lo in ((E, j0[g] - n), (O, j0[g] - n - 1)):
                        for t in range(C2):
                            v = uhalves(X[g][t])
                            keep = [lo <= s <= m - i0[g] for s in (t, t + C2)]
                            X[g][t] = umk(*(h if k else DEAD for h, k in zip(v, keep)))
        left -= 1
        if left == 0:  # the latest the kernel lifts
            stats["lift"] += 1
            left = period
            for X in (E, O):
                for row in X:
                    row[:] = [max_s(v, DEAD2) for v in row]
        if budget < 1:
            budget = margin()
