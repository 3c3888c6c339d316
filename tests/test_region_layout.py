"""Shared-memory and record indexing of the register-path step instances and of
the row-parallel adjoint, in the layout they have now: the sizes come from the
library's own header (csrc/sfd_types.h, compiled for the host) and the field
offsets and cell counts from the kernels' source, so that a change on either
side is compared with the other.  Every address that any lane forms for a grid,
transfer addresses of both grids included, lies inside the string's region (and
so inside what warp_smem_floats makes the launch ask for), and no two cells of
a layout coincide."""

import os
import re
import shutil
import subprocess

import numpy as np
import pytest

WARP = 32
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_18505_gb300", "csrc")
STEP = open(os.path.join(CSRC, "sfd_step_reg.cuh")).read()
KERNEL = open(os.path.join(CSRC, "sfd_kernel.cu")).read()

PROGRAM = """
#include <cstdio>
#define __host__
#define __device__
#include "sfd_types.h"
int main() {
  std::printf("static %d\\n", sfd::kStaticSmemBytes);
  for (int mu = 1; mu <= 9; mu += 2)
    for (int mz = 0; mz <= 145; mz += mz ? 2 : 1)
      for (int zj = 0; zj < 2; ++zj)
        std::printf("region %d %d %d %d\\n", mu, mz, zj, sfd::warp_smem_floats(mu, mz, zj));
  for (int nu = 1; nu <= sfd::kAdjRowsMax; nu += 2)
    for (int nz = 0; nz < 600; nz += 7) std::printf("rows %d %d %d\\n", nu, nz, sfd::adj_rows_smem_bytes(nu, nz));
}
"""


@pytest.fixture(scope="module")
def header(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("types")
    (d / "main.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "sizes")], check=True)
    out = {}
    for line in subprocess.run([str(d / "sizes")], capture_output=True, text=True, check=True).stdout.splitlines():
        key, *v = line.split()
        out[(key, *map(int, v[:-1]))] = int(v[-1])
    return out


def constant(pattern, src=STEP):
    m = re.findall(pattern, src)
    assert len(m) == 1, pattern
    return m[0]


RECORD = int(constant(r"constexpr int kRec = (\d+);"))
FIELDS = {records: int(n) for records, n in zip((True, False), constant(r"p \+= \(kRecs \? (\d+) : (\d+)\) \* RZ;"))}
# field numbers by name: as in "oSX0 = 6 * kFld", those of the right-hand side's slots by layout
FIELD = {m[0]: int(m[1]) for m in re.findall(r"\b(o[A-Z]+\d?) = (\d+) \* kFld", STEP)}
FIELD.update(oZ=0, oDZ=1)
SV = {True: ("oSF0", "oSF1"), False: tuple(int(n) for n in constant(r"oSV0 = kRecs \? oSF0 : (\d+) \* kFld, oSV1 = kRecs \? oSF1 : (\d+) \* kFld"))}


def rows_per_lane(n):
    """Odd m with 32 m >= n + 1 (host rule of sfd_api.cu)."""
    return max(1, (n + WARP) // WARP) | 1


def instance(m_z, folded, warps):
    """What run_job_exc picks: (layout, warps that step the string)."""
    if not folded:
        return "factored", 1
    warps = warps if m_z >= warps else 1
    if m_z in (1, 3):
        return "arrays", 1
    return "records", warps


def check_grid(header, n_t, n_l, folded, warps):
    n_u, n_z = n_t - 1, n_l - 1
    m_u, m_z = rows_per_lane(n_u), rows_per_lane(n_z)
    if m_u > 9 or ("region", m_u, m_z, int(folded)) not in header:
        return 0
    layout, ng = instance(m_z, folded, warps)
    region = 4 * header[("region", m_u, m_z, int(folded))]      # bytes
    slots = 4 * 2 * (WARP * m_u + 4)                            # the two transverse slots come first
    records = layout == "records"
    row_bytes = RECORD if records else 4
    cells = WARP * m_z + 4                                      # of one field
    fld = 4 if records else 4 * cells
    n_fields = 16 if layout == "factored" else FIELDS[records]
    base = slots + 2 * row_bytes

    def at(field, rows):   # addresses of a field, inside the region and inside the field's own cells
        rows = np.asarray(rows)
        number = FIELD.get(field, field)
        assert 0 <= number < n_fields, field
        assert rows.min() >= -2 and rows.max() < cells - 2, (field, rows.min(), rows.max())
        a = base + row_bytes * rows + fld * number
        assert a.min() >= slots and a.max() + 4 <= region, (field, n_t, n_l, layout)
        return a

    # fields apart: a field's cells are fld apart (arrays) or words of one record
    assert fld * n_fields <= RECORD if records else fld >= 4 * cells
    # every longitudinal row has one owner among the warps
    owned = np.concatenate([lane + WARP * np.arange(pw, m_z, ng)[:, None] for pw in range(ng)
                            for lane in [np.arange(WARP)[None]]]).ravel()
    assert np.array_equal(np.sort(owned), np.arange(WARP * m_z))
    rows = np.arange(WARP * m_z)
    for f in ("oZ", "oDZ", "oAZ", "oXZ"):                       # own value and both neighbours
        at(f, rows - 1), at(f, rows), at(f, rows + 1)
    if records:                                                 # right-hand side, spare accelerations and responses
        at("oRZ", rows)
        for f in ("oE2", "oE3"):
            at(f, rows - 1), at(f, rows + 1)
    # transfer: the map of rows -1 .. MU of every lane (pad rows point at node N_l + 1)
    i = np.arange(-1, WARP * m_u + 1)
    pos = (i + 1) * n_l
    mm = np.where(i < n_u, pos // n_t, n_l + 1)
    for f in ("oZ", "oAZ", "oXZ") + (("oE2", "oE3") if records else ()):
        at(f, mm - 1), at(f, mm)                                # interpolated to the rows
    real = mm[(i >= 0) & (i < n_u)]
    for s0, s1 in (("oSF0", "oSF1"), ("oSX0", "oSX1"), SV[layout != "arrays"]):
        at(s0, real), at(s1, real + 1)                          # sums stored by an interval's last row
        at(s0, rows + 1), at(s1, rows + 1)                      # ... and read by the longitudinal rows
    return 1


def test_every_access_lies_in_the_region(header):
    checked = 0
    for n_t in list(range(2, 289, 5)) + [32, 33, 96, 97, 160, 161, 224, 225, 256, 288]:
        for n_l in sorted({2, 3, 32, 33, 96, 97, 160, 161, 384, 385, 768, 769, max(2, n_t // 3), n_t, n_t + 1,
                           2 * n_t, 4 * n_t + 3, 16 * n_t}):
            for folded, warps in ((True, 1), (True, 4), (True, 8), (False, 1)):
                checked += check_grid(header, n_t, n_l, folded, warps)
    assert checked > 3000


def test_register_rows_of_a_group():
    """A group's warp holds three longitudinal rows in registers: the instances
    403 and 803 are taken only where that covers every row."""
    for warps, code, most in ((4, 403, 12), (8, 803, 24)):
        cond = constant(r"g\.ng == %d && ([^)]*)\) step_string<MU, %d," % (warps, code))
        assert re.search(r"m_z <= %d" % most, cond) and most == 3 * warps


def test_exchange_cells(header):
    """The warps of a group exchange four maxima per lane: float4 cell
    buffer * 32 ng + warp * 32 + lane, two buffers."""
    cells = int(constant(r"float xcells\[(\d+)\];", KERNEL))
    for ng in (4, 8):
        idx = [b * 32 * ng + pw * 32 + lane for b in (0, 1) for pw in range(ng) for lane in range(WARP)]
        assert len(set(idx)) == len(idx) and 4 * (max(idx) + 1) <= cells
    job_cells = int(constant(r"__shared__ int jcell\[(\d+)\];", KERNEL))
    assert 4 * cells + 4 * job_cells <= header[("static",)]


def test_adjoint_rows_sizes(header):
    """What the row-parallel adjoint carves (arrays counted in its source)
    against adj_rows_smem_bytes, and the trajectory records it copies 16 bytes
    at a time against the forward's stride."""
    src = open(os.path.join(CSRC, "sfd_adjoint_rows.cu")).read()
    carve = src[src.index("int* ROW0 = nullptr") - 3000:src.index("const int n = static_cast<int>(pf - recs);")]
    n_du, n_dz = len(re.findall(r"= du\(\)", carve)), len(re.findall(r"= dz\(\)", carve))
    more = carve.count("pd += (kZLev - 1) * zl;")
    lev = int(constant(r"constexpr int kAdjRowsLev = (\d+);", open(os.path.join(CSRC, "sfd_types.h")).read()))
    zlev = int(constant(r"constexpr int kAdjRowsZLev = (\d+);", open(os.path.join(CSRC, "sfd_types.h")).read()))
    for key, got in header.items():
        if key[0] != "rows":
            continue
        n_u, n_z = key[1:]
        stride = -(-(2 * n_u + 2 * n_z + 2) // 4) * 4
        ru, rz = n_u + 4, n_z + 4
        want = 4 * 3 * stride + 8 * n_du * ru + 8 * 2 * lev * n_u + 4 * ru
        if n_z:
            want += 8 * (n_dz + more * (zlev - 1)) * rz + 4 * 2 * rz
        assert got == want, key
