"""One-token steps on both sides of the lines between the kernel merged by clusters and the streaming kernel."""
import pytest
import torch

from paper_2510_18546_b200 import enl, synth
from tests.helpers import Session, check_close

pytestmark = pytest.mark.gpu


def check_step(hq, hkv, d, lens, episodes, want_mass, ctas, what):
    """The step is right, and its splits are the `ctas` CTAs of a cluster (or, with None, any other number: the streaming kernel's)."""
    wl = synth.make_small(81, 1, hq, hkv, d, [lens] * episodes, [list(range(len(lens)))] * episodes, [1] * episodes, [1] * episodes, name=what)
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        out, mass, _ = s.attend(0, q, kn, vn, want_mass=want_mass)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        p = enl.enl_plan_inspect(s.cache)
        assert p["merge_kind"] == 3
        if ctas is None:
            assert p["n_splits"] not in (1, 2, 4, 8, 16)
        else:
            assert p["n_splits"] == ctas
        for b in range(episodes):
            ro, rm, _ = s.oracle(0, b, q[b:b + 1], kn[b:b + 1], vn[b:b + 1])
            check_close(out[b:b + 1], ro, mass[b:b + 1] if want_mass else None, rm if want_mass else None, what=what)


# (q heads, kv heads, head_dim, pages per CTA at the line, CTAs per cluster, episodes)
LINES = [(32, 8, 128, 64, 16, 1), (8, 2, 128, 88, 16, 1), (32, 8, 64, 112, 16, 1), (16, 8, 128, 88, 8, 2)]


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("above", [False, True])
@pytest.mark.parametrize("line", LINES)
def test_step_at_the_line(line, above, want_mass):
    hq, hkv, d, pages, ctas, n = line
    # cached pages: a multiple of eight, as they are counted; the new token has one of its own
    cached = pages * ctas + (8 if above else -16)
    lens = [16 * (cached // 3), 16 * (cached - cached // 3 - 7), 100]
    check_step(hq, hkv, d, lens, n, want_mass, None if above else ctas, f"line {line}")


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("pages", [70, 72, 76])
def test_lists_of_two_ctas_per_sm(pages, want_mass):
    """Thirty-two streams of many groups, in clusters of eight as long as two of their CTAs fit a multiprocessor."""
    cached = 8 * pages - 8
    check_step(16, 2, 128, [16 * 5] * (cached // 5) + [16 * (cached % 5)], 16, want_mass, 8, f"{pages} pages")
