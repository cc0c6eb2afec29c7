"""Contexts share a page of error words: a run that is not finite is reported by its
own context alone, and a word that comes back is clean for the next context, also
beyond the page's 1024 words."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _context(ns, stream=None):
    return ns.ns_init([dict(n=8, nu=0.0, dt=1e-3)], ns.NS_FP32, stream)


def _status(ns, ctx):
    try:
        ns.ns_sync(ctx)
    except ns.NsError as e:
        return e.status
    return 0


def _spoil(ns, ctx):
    a = np.zeros((3, 8, 8, 5), dtype=np.complex128)
    a[0, 1, 0, 0] = np.nan
    ns.ns_set_state(ctx, 0, a)
    ns.ns_step(ctx, 1)


@pytest.mark.parametrize("count", [3, 1030])
def test_words_of_live_and_later_contexts(ns, count):
    live = [_context(ns) for _ in range(count)]
    try:
        bad = {0, 1, count - 1}
        for i in bad:
            _spoil(ns, live[i])
        assert [i for i in range(count) if _status(ns, live[i]) == ns.NS_ERR_NONFINITE] == sorted(bad)
    finally:
        for c in live:
            ns.ns_destroy(c)
    for _ in range(3):
        c = _context(ns)
        try:
            ns.ns_step(c, 1)
            assert _status(ns, c) == 0
        finally:
            ns.ns_destroy(c)
