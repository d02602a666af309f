"""max_workspace_bytes and workspace_bytes against the device memory that contexts really take.

Many contexts of the smallest system, so that what each one owns beyond its count adds up.  The
allocator hands out memory in blocks of 2 MB shared by small allocations; a handful of those is the slack.
"""
import pytest

import rix_inputs as ri

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_10343_gb300.rix import Exchange, RixError  # noqa: E402

N = 48
SLACK = 8 << 20


def _taken(s, **kw):
    """Device memory taken by N contexts, and their workspace_bytes."""
    Exchange.from_system(s, **kw).close()  # modules and pools are loaded
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ex = [Exchange.from_system(s, **kw) for _ in range(N)]
    taken = free - torch.cuda.mem_get_info()[0]
    owned = [e.stats()["workspace_bytes"] for e in ex]
    for e in ex:
        e.close()
    return taken, owned


@pytest.fixture(scope="module")
def one():
    return ri.water_cluster(1, 5, cutoff=False)


def test_workspace_bytes_is_the_memory_owned(one):
    taken, owned = _taken(one)
    assert taken <= sum(owned) + SLACK


def test_limit_bounds_the_memory_owned(one):
    limit = 960 << 10  # the system's arrays take 864 KB
    taken, owned = _taken(one, max_workspace_bytes=limit)
    assert max(owned) <= limit
    assert taken <= N * limit + SLACK


def test_limit_of_what_a_context_needs_is_enough(one):
    # the arrays alone, as a context under a limit takes them, and one byte less
    need = Exchange.from_system(one, max_workspace_bytes=1 << 30)
    w = need.stats()["workspace_bytes"]
    need.close()
    free = Exchange.from_system(one)
    assert free.stats()["workspace_bytes"] >= w
    free.close()
    with pytest.raises(RixError):
        Exchange.from_system(one, max_workspace_bytes=w // 2)
