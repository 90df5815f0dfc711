"""The barrier protocol of k_pn_gram over items of different, odd and even, numbers of stages, on the CPU: stage and window
counters run on across items, the two groups of A warps take alternate stages of that running count, an item's last window may
be one stage long, and the issuers and the drain warps carry their window parity over.  The model of test_chi0_protocol with
the items' lengths as a list: every wait must pass only after its event, no stage may be overwritten under its MMAs, and at the
end (also after waits that gave up) no copy and no MMA is in flight."""
import random

import pytest

from tests.test_chi0_panels_protocol import _constant
from tests.test_chi0_protocol import _Bar


def _run_items(items, nstage, promote, seed, timeouts=False, withhold=False, wpg=4, ndrain=3):
    rnd = random.Random(seed)
    nb = 2 * nstage
    full_b, full_a = [_Bar(1) for _ in range(nb)], [_Bar(wpg) for _ in range(nb)]
    empty, acc_full, drained = [_Bar(1) for _ in range(nstage)], [_Bar(1), _Bar(1)], [_Bar(ndrain), _Bar(ndrain)]
    done_bar = _Bar(2)
    windows, gs = [], 0                           # running stages of every window
    for n in items:
        windows += [list(range(gs + i, gs + min(i + promote, n))) for i in range(0, n, promote)]
        gs += n
    total = gs
    landed, formed, done, drains = set(), {}, set(), {}
    copies, mmas, errors, abort = [], [], [], [False]

    def wait(bar, parity, event, what, honour=True):
        spins = 0
        while not bar.passes(parity):
            if honour and abort[0]:
                return False
            spins += 1
            if honour and timeouts and spins > 8 and rnd.random() < 0.01:
                abort[0] = True
                return False
            yield
        if not event():
            errors.append("early pass: " + what)
        return True

    def producer():
        sent = 0
        for g in range(0 if withhold else total):
            if not (yield from wait(empty[g % nstage], (g // nstage) & 1 ^ 1, lambda: g < nstage or g - nstage in done, f"free {g}")):
                break
            copies.append(g)
            sent = g + 1
        for g in range(max(0, sent - nstage), sent):
            yield from wait(full_b[g % nb], (g // nb) & 1, lambda: g in landed, f"copy {g}", honour=False)
        if copies:
            errors.append("producer left with copies in flight")

    def a_warp(group):
        for g in range(group, total, 2):
            if not (yield from wait(full_b[g % nb], (g // nb) & 1, lambda: g in landed, f"copy {g}")):
                return
            if g >= nstage and g - nstage not in done:
                errors.append(f"A tile {g} overwritten under its MMAs")
            formed[g] = formed.get(g, 0) + 1
            full_a[g % nb].arrive()

    def issuer(par):
        ok = True
        for w in range(par, len(windows), 2):
            if w >= 2:
                ok = yield from wait(drained[par], ((w - 2) >> 1) & 1, lambda: drains.get(w - 2, 0) == ndrain, f"buffer {w}")
            for g in windows[w] if ok else []:
                ok = yield from wait(full_a[g % nb], (g // nb) & 1, lambda: formed.get(g, 0) == wpg, f"A tile {g}")
                if not ok:
                    break
                mmas.append((g, empty[g % nstage]))
                yield
            if not ok:
                break
            mmas.append((("window", w), acc_full[par]))
        mmas.append((("last", par), done_bar))
        yield from wait(done_bar, 0, lambda: {("last", 0), ("last", 1)} <= done, "every MMA finished", honour=False)

    def drain_warp():
        for w in range(len(windows)):
            if not (yield from wait(acc_full[w & 1], (w >> 1) & 1, lambda: ("window", w) in done, f"window {w}")):
                return
            drains[w] = drains.get(w, 0) + 1
            drained[w & 1].arrive()

    actors = [producer(), issuer(0), issuer(1)] + [a_warp(i % 2) for i in range(2 * wpg)] + [drain_warp() for _ in range(ndrain)]
    for _ in range(1000000):
        if not actors:
            if mmas:
                errors.append("TMEM freed with MMAs in flight")
            if not abort[0] and (len(formed) != total or len(drains) != len(windows)):
                errors.append("work missing without an abort")
            return errors, abort[0]
        r = rnd.random()
        if r < 0.15 and copies:
            g = copies.pop(rnd.randrange(len(copies)))
            landed.add(g)
            full_b[g % nb].arrive()
        elif r < 0.3 and mmas:
            key, bar = mmas.pop(0)
            done.add(key)
            bar.arrive()
        else:
            a = rnd.choice(actors)
            try:
                next(a)
            except StopIteration:
                actors.remove(a)
    return errors + ["no progress"], None


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("items", [[1] * 9, [3, 1, 5, 1, 1, 7], [15, 2, 1, 8, 3], [5, 5, 5, 5], [128, 1, 33]])
@pytest.mark.parametrize("fault", [{}, {"timeouts": True}, {"withhold": True, "timeouts": True}])
def test_items_of_any_number_of_stages(items, extra, fault):
    for seed in range(4):
        errors, aborted = _run_items(items, _constant("PG_NSTAGE") + extra, _constant("PG_PROMOTE"), seed, **fault)
        assert not errors, (items, seed, errors[:3])
        assert bool(aborted) <= bool(fault) and (aborted or not fault.get("withhold"))


def test_a_ring_shorter_than_the_windows_is_caught():
    assert any(_run_items([9, 3, 5], 2, 4, seed)[0] for seed in range(10))
