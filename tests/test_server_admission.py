"""Which jobs the request loop refuses at submit by their device bytes (no GPU needed)."""
import pytest

import workloads as w

from .test_server_host import _system, ll  # noqa: F401  (ll: the fixture)


def test_a_job_that_fits_the_budget_is_accepted(ll):  # noqa: F811
    """A job is refused by the bytes it is admitted with (its spheres' columns on the grid its
    orbitals are transformed on), not by ll_footprint's bound, which reads no Miller index."""
    b = w.get_bundle(w.config_small())
    bound = ll.footprint(**_system(b))
    srv = ll.Server(hbm_budget_bytes=int(0.75 * bound), max_slots=1)
    srv.cancel(srv.submit(20, None, 0.1, **_system(b)))
    srv.close()
    srv = ll.Server(hbm_budget_bytes=int(0.1 * bound), max_slots=1)
    with pytest.raises(ll.LLError) as e:
        srv.submit(20, None, 0.1, **_system(b))
    assert e.value.code == ll.LL_ENOMEM and "budget" in str(e.value)
    srv.close()
