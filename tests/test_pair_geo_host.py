"""The geometry every pass is launched with (``PairGeo`` in
``csrc/fock_kernels.cuh``, ``PersistGeo`` in ``csrc/fock_persist.cuh``), printed by a
host program from the kernels' headers, against what its launches and index maps
rely on, for the users' grid sizes and the plans' working grids (CPU; no GPU):

* the factors of both kinds of stage multiply to N, and the block passes to 4 M;
* CTAs are whole warps of at most 1024 threads, the column pass's of whole lines;
* shared memory fits a CTA, and as many CTAs as a launch bound asks for fit an SM
  with at least 40 registers a thread;
* the places of frequencies and rows are permutations;
* the one-launch kernels' threads and shared memory cover every size they run.
"""

import subprocess

import pytest

from tests._common import host_program

SMEM_PER_SM, SMEM_PER_CTA, RESERVED = 233472, 232448, 1024
USER = {8, 12, 16, 24, 32, 36, 48, 64, 72, 96}
PAIR = {20, 28, 40, 56, 60, 80}
ONE_LAUNCH = {20, 24, 28, 32, 40, 48, 56, 60, 64, 72, 80, 96}
KEYS = ("type", "N", "tile", "user", "A", "B", "CA", "CB", "block", "thr_plane", "thr_col", "smem_plane", "smem_col",
        "min_plane", "min_col", "np", "cbytes")


@pytest.fixture(scope="module")
def printed(tmp_path_factory):
    exe = host_program("pair_geo_driver.cu", tmp_path_factory.mktemp("pair_geo"),
                       extra=("-gencode", "arch=compute_103a,code=sm_103a"))
    geo, persist = [], {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        w = line.split()
        v = [int(x) for x in w[1:]]
        if w[0] == "persist":
            persist[v[0]] = v[1:]
            continue
        g = dict(zip(KEYS, v))
        rest, n = v[len(KEYS):], g["N"]
        g.update(rows=rest[:n], cols=rest[n:2 * n], back=rest[2 * n:])
        assert len(rest) == 3 * n
        geo.append(g)
    return geo, persist


def test_every_size_and_tiling_is_listed(printed):
    geo, _ = printed
    for t in (0, 1, 2):
        assert {g["N"] for g in geo if g["type"] == t and g["tile"] == 0 and g["user"]} == USER
        assert {g["N"] for g in geo if g["type"] == t and g["tile"] == 0 and not g["user"]} == PAIR
        assert {g["N"] for g in geo if g["type"] == t and g["tile"] == 1} == (set() if t == 2 else {16, 96})


def test_factors_and_places(printed):
    for g in printed[0]:
        n = g["N"]
        assert g["A"] * g["B"] == n and g["CA"] * g["CB"] == n, g
        assert g["block"] == (g["type"] == 1 and g["tile"] == 0) and n % 4 == 0, g
        assert sorted(g["rows"]) == list(range(n)) and sorted(g["cols"]) == list(range(n)), g
        assert g["back"] == list(range(n)), g  # row_of undoes place_of_row


def test_ctas_and_shared_memory(printed):
    for g in printed[0]:
        assert g["thr_plane"] % 32 == 0 and g["thr_plane"] <= 1024, g
        assert g["thr_col"] % (2 * g["np"]) == 0 and g["thr_col"] <= 1024, g
        assert max(g["smem_plane"], g["smem_col"]) <= SMEM_PER_CTA, g
        if g["block"]:
            assert g["thr_plane"] >= 4 * g["N"], g  # an item of the row stage a thread
        for m, thr, smem in ((g["min_plane"], g["thr_plane"], g["smem_plane"]),
                             (g["min_col"], g["thr_col"], g["smem_col"])):
            assert 1 <= m <= 32 and m * thr <= 2048, g
            assert m * (smem + RESERVED) <= SMEM_PER_SM and 65536 // (m * thr) >= 40, g


def test_the_one_launch_kernels_cover_their_sizes(printed):
    geo, persist = printed
    for t, (threads, smem, ctas) in persist.items():
        assert threads % 32 == 0 and ctas * (smem + RESERVED) <= SMEM_PER_SM
        for g in geo:
            if g["type"] == t and g["tile"] == 0 and g["N"] in ONE_LAUNCH:
                assert threads % (2 * g["np"]) == 0 and smem >= max(g["smem_plane"], g["smem_col"]), g
                if g["block"]:
                    assert threads >= 4 * g["N"], g
