"""Host set-up of a solve's sources (eik_host.h), compiled for the host: the device tables of the fixed nodes fit the room
that is allocated for them, whichever layout the sources have."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "eik_host.h"
extern "C" int tables(int n, const double* xyz, int nx, int ny, int nz, int elem, long long* out) {
    const eikh::Bricks g{(nx + 7) / 8, (ny + 7) / 8, (nz + 7) / 8, 0};
    std::vector<eikh::Cand> cand;
    eikh::source_candidates(xyz, n, nx, ny, nz, 1.0, g, cand);
    const std::vector<double> r(cand.size(), 1.0);
    const std::vector<eikh::FixNode> fix = eikh::fixed_nodes(cand, r, 1.0);
    std::vector<int32_t> sb, enq;
    eikh::first_active(fix, g, sb, enq);
    const std::vector<int32_t> genq = eikh::groups_of(enq, g, (g.BX + 1) / 2, (g.BY + 1) / 2, 0);
    const eikh::SolveTables t = eikh::solve_tables(cand.size(), fix.size(), sb.size(), enq.size(), genq.size(), elem);
    const size_t at[10] = {t.cand_b, t.cand_p, t.fix_b, t.fix_p, t.fix_v, t.src_b, t.enq, t.genq, t.saved, t.end};
    const size_t len[9] = {4 * cand.size(), 4 * cand.size(), 4 * fix.size(), 4 * fix.size(), 8 * fix.size(),
                           4 * sb.size(), 4 * enq.size(), 4 * genq.size(), elem * fix.size()};
    for (int i = 0; i < 9; ++i)
        if (at[i] % 256 || at[i] + len[i] > at[i + 1]) return 1 + i;
    out[0] = static_cast<long long>(t.end);
    out[1] = static_cast<long long>(eikh::solve_tables_room(cand.size(), elem));
    out[2] = static_cast<long long>(fix.size());
    out[3] = static_cast<long long>(enq.size());
    out[4] = static_cast<long long>(genq.size());
    return 0;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_setup")
    src, lib = d / "harness.cpp", d / "harness.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1811_00009_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    return C.CDLL(str(lib))


@pytest.mark.parametrize("elem", [4, 8])
@pytest.mark.parametrize("kind", ["none", "one", "spread corners", "low corners", "in cells", "same node"])
def test_tables_fit_their_room(host, kind, elem):
    n = 257
    corners = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), -1).reshape(-1, 3)
    rng = np.random.default_rng(3)
    xyz = {"none": np.zeros((0, 3)), "one": np.array([[16.0, 16.0, 16.0]]), "spread corners": 32.0 * corners + 16.0,
           "low corners": 8.0 * corners, "in cells": rng.uniform(0, n - 1, (700, 3)),
           "same node": np.full((600, 3), 24.0)}[kind]
    xyz = np.ascontiguousarray(xyz)
    out = (C.c_longlong * 5)()
    rc = host.tables(len(xyz), xyz.ctypes.data_as(C.POINTER(C.c_double)), n, n, n, elem, out)
    assert rc == 0
    end, room, nfix, nenq, ngenq = out
    assert end <= room
    if kind == "spread corners":                 # every source activates four bricks, in four groups
        assert (nfix, nenq, ngenq) == (512, 2048, 2048)
