"""Shared-memory layout of the register-path step instances, modelled on the
CPU (csrc/sfd_step_reg.cuh, step_string): every field access of every lane
lies inside the region the host allots a string (warp_smem_floats) and the
fields do not overlap, for the instances that keep longitudinal rows in
registers (one array per field; groups of 4 and 8 warps: records) and for
those that keep them in records."""

import pytest

WARP = 32


def region_bytes(m_u, m_z):
    """warp_smem_floats of sfd_types.h, folded longitudinal matrix."""
    return 4 * (2 * (WARP * m_u + 4) + 12 * (WARP * m_z + 4))


def addresses(m_u, m_z, ng, kind):
    """(address, field, row) of every field of every row the instance touches,
    in bytes from the region's start."""
    records = kind != "arrays"
    row_bytes = 44 if records else 4
    fld = 4 if records else 4 * (WARP * m_z + 4)
    base = 4 * 2 * (WARP * m_u + 4) + 2 * row_bytes
    n_fields = 11 if records else 10
    rows = set()
    for pw in range(ng):
        mine = range(pw, m_z, ng)
        if kind == "group":   # three registers per warp, missing rows read the first one's
            ks = [k if k < m_z else pw for k in (pw, pw + ng, pw + 2 * ng)]
            assert set(mine) <= set(ks)
        else:                 # batches of up to four, a short one repeats its last row
            ks = list(mine)
        rows |= {lane + WARP * k for k in ks for lane in range(WARP)}
    assert rows == set(range(WARP * m_z))   # every row has an owner
    rows |= {r + d for r in rows for d in (-1, 1)}          # neighbours, transfer slots of node row + 1
    rows |= {-1, WARP * m_z + 1}                            # a map's nodes m - 1 >= -1 and m + 1 <= n_z + 2
    return [(base + row_bytes * r + fld * f, f, r) for r in rows for f in range(n_fields)]


@pytest.mark.parametrize("m_u", [1, 3, 5, 7, 9])
def test_fields_lie_in_the_region_and_apart(m_u):
    cases = [(1, 1, "arrays"), (3, 1, "arrays")]
    cases += [(m, ng, "records") for m in (5, 7, 9, 25, 53) for ng in (1, 2, 4, 8)]
    cases += [(m, 4, "group") for m in (5, 7, 9, 11)] + [(m, 8, "group") for m in (13, 15, 23)]
    for m_z, ng, kind in cases:
        acc = addresses(m_u, m_z, ng, kind)
        low = 4 * 2 * (WARP * m_u + 4)
        assert min(a for a, _, _ in acc) >= low, (m_z, ng, kind)
        assert max(a for a, _, _ in acc) + 4 <= region_bytes(m_u, m_z), (m_z, ng, kind)
        where = {}
        for a, f, r in acc:
            assert a % 4 == 0 and where.setdefault(a, (f, r)) == (f, r), (m_z, ng, kind)


def test_adjoint_rows_fit_what_the_host_allots():
    """adj_rows_smem_bytes of sfd_types.h against the carving of
    sfd_adjoint_rows.cu (bytes), and the rows each array is indexed by."""
    for n_u in (1, 2, 31, 100, 255):
        for n_z in (0, 1, 31, 143, 800):
            rec = (2 * n_u + 2 * n_z + 2 + 3) // 4 * 4
            ru, rz = n_u + 4, (n_z + 4 if n_z else 0)
            host = 4 * (3 * rec + 28 * ru + 4 * 8 * n_u + 36 * rz + ru + 2 * rz)
            carved = 4 * 3 * rec                    # records
            carved += 8 * 14 * ru                   # FA FC FR (2 each), X XP P0 P1 Q0 Q1 TN TX
            carved += 8 * 18 * rz                   # NZ XZ RZ LZ LDZ BZ NZP XZP, E and G (2 each), KA KC (3 levels each)
            carved += 8 * 2 * 8 * n_u               # reduction weights
            carved += 4 * ru + 4 * 2 * rz           # A, AZ, ROW0
            assert carved == host
            assert 2 + n_u - 1 + 2 < ru             # X[i + 2] of the last row, two cells at either end
            if n_z:
                assert n_z + 2 < rz                 # ROW0[m], m <= n_l + 1 = n_z + 2
