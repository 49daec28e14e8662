"""The device memory of a context, field by field: a workspace limit that admits
it has to go on admitting it."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,nt", [((32, 24, 20), 4), ((45, 8, 50), 3)])
def test_workspace_of_a_context(shape, nt):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_12820_gb300 import claire as C
    n1, n2, n3 = shape
    N = n1 * n2 * n3
    p3 = (n3 // 2 + 1 + 3) // 4 * 4                                   # padded half spectrum
    tiles = -(-n3 // 32) * (-(-n2 // 8)) * (-(-n1 // 4))
    # m0, m1, v, X-, X+, div v, c, mt, scratch (3 + 1 + 1), forward X-: 22 fields;
    # m^j, grad m^j, l^j: 5 per level
    full = 4 * N * (22 + 5 * (nt + 1)) + 8 * 3 * n1 * n2 * p3
    full += 8 * (4 * 1216 + 16) + 4 + 4 * 16 * tiles                  # reductions, flag, box entries
    try:
        C.set_workspace_limit(full)
        with C.Registration(shape, nt, 1e-2, 1.0) as reg:
            assert reg.workspace_bytes() == full
    finally:
        C.set_workspace_limit(0)
