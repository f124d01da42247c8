"""The hand-overs between the roles of an attention CTA (csrc/wk_attention.cu) under all kinds of timing.  The roles themselves are
compiled for the host, with barriers, copies and matrix products that the schedule completes; every role in turn is held at each of
its barrier operations until nothing else can move, which is the longest that any delay can last."""
import ctypes as C
import os
import re
import shutil
import subprocess

import pytest

from paper_2605_22718_b200.build import CSRC, ROOT, _nvcc

HOST = os.path.join(ROOT, "tests", "host")


def roles_source():
    src = open(os.path.join(CSRC, "wk_attention.cu")).read()
    cut = re.search(r"template <[^>]*>\n__global__", src).start()
    init = re.search(r"if \(tid == 0\) \{\n(.*?)fence_mbar_init", src[cut:], re.S).group(1)
    body = src[:cut].replace('#include "ptx_sm100.cuh"\n', "")
    for name in ("bool wait_or_abort(", "float fmax3(", "float fmax3_nan("):   # PTX through and through: stand-ins
        assert name in body
        body = body.replace(name, name[:-1] + "_ptx(", 1)
    warp_wide = "__device__ __forceinline__ int count_tiles("                  # its lanes work on different slots
    assert warp_wide in body
    body = body.replace(warp_wide, "int count_tiles(const AttnParams& p, int tb, int te);\n" + warp_wide[:-1] + "_of_a_warp(", 1)
    body = re.sub(r"\basm(\s+volatile)?\s*\(", "WK_ASM(", body)
    return body + "template <int kKv> void init_barriers(CtaShared<kKv>& sh) {\n  constexpr bool kLse = is_lse<kKv>;\n" + init + "}\n"


@pytest.fixture(scope="module", params=[80, 64, 128], ids=["tiles_of_80", "tiles_of_64", "lse_only"])
def run(request, tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    out = tmp_path_factory.mktemp("roles")
    (out / "roles.inc").write_text(roles_source())
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    lib = str(out / "libroles.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-DWK_TEST_ROWS={request.param}",
                    "-I", str(out), "-I", cuda, "-I", CSRC, os.path.join(HOST, "attention_roles.cc"), "-o", lib], check=True)
    fn = C.CDLL(lib).run_roles

    def call(H, lq, segs, slots, C_rows, n_full, n_ranges, grid, schedules=20, hold=True):
        what = C.create_string_buffer(400)
        bad = fn(H, lq, (C.c_int * len(segs))(*segs), len(segs), (C.c_int * len(slots))(*slots), len(slots), C_rows, n_full, n_ranges,
                 grid, schedules, int(hold), what, 400)
        assert not bad, what.value.decode()
    call.lse_only = request.param == 128
    return call


# One Q tile (lq <= 128, or the last pair of 257 .. 384 rows) or two; several units on a CTA; pieces of one tile, two, and more than
# there are stages; slots that are stale (odd) or holes, so that a piece has no tile at all.
@pytest.mark.parametrize("lq", [100, 200, 300])
@pytest.mark.parametrize("segs,slots,rows", [((60,), (), 8), ((100,), (), 8), ((60, 130, 33), (), 8), ((500,), (), 8),
                                             ((70,), (2, 1, 0), 100), ((), (1, 3), 40), ((), (4, -1), 90)])
def test_units_one_after_another(run, lq, segs, slots, rows):
    if run.lse_only:
        slots, segs = slots or (0, 2), ()
    H = 2
    units = H * ((lq + 255) // 256) * (len(slots) if run.lse_only else 1)
    run(H, lq, segs, slots, rows, units, 0, 1)


@pytest.mark.parametrize("lq", [100, 300])
@pytest.mark.parametrize("ranges", [2, 3, 5])
@pytest.mark.parametrize("n_full", [0, 1])
def test_ranges_that_cross_units(run, lq, ranges, n_full):
    """The walk of a CTA: a whole unit where there is one, units inside its range, and the piece of the unit it starts in."""
    if run.lse_only:
        pytest.skip("whole units only")
    run(3, lq, (200, 90), (0, 1), 70, n_full, ranges, ranges, schedules=10)
