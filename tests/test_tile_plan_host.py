"""The choice of register tiles (plan_tiles of cx_tile.cu) is host arithmetic:
for every size, scheme and call length it ends, on any machine, and gives
tiles that cover the grid and keep at least half of their cells."""
import subprocess
import sys

# in a process of its own: a division by zero ends the process on x86
SCRIPT = r"""
import ctypes as C
from paper_1301_5058_gb300 import _build
_build.build()
import paper_1301_5058_gb300 as cx

class Grid(C.Structure):
    _fields_ = [("nx", C.c_int), ("ny", C.c_int), ("count", C.c_int)]

class Plan(C.Structure):
    _fields_ = [("steps", C.c_int), ("lx", C.c_int), ("r", C.c_int), ("threads", C.c_int),
                ("heun", C.c_bool)]

# double cx::plan_tiles(const TileGrid *, int, int, bool, bool, long long, TilePlan *)
plan_tiles = cx.lib()._ZN2cx10plan_tilesEPKNS_8TileGridEiibbxPNS_8TilePlanE
plan_tiles.restype = C.c_double
plan_tiles.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_bool, C.c_bool, C.c_longlong, C.c_void_p]
SIDES = (1, 15, 16, 17, 33, 64, 129, 256, 1021, 2048, 16384, 1000000)
sizes = [(nx, ny) for nx in SIDES for ny in SIDES if nx * ny <= 1 << 28]
for heun in (False, True):
    for per_step in (False, True):
        for steps in (1, 2, 3, 4, 7, 8, 9, 16, 23, 64, 1000, 1 << 40):
            for mix in [[z] for z in sizes] + [sizes[i::37] for i in range(37)]:
                grids = (Grid * len(mix))(*[Grid(nx, ny, 1) for nx, ny in mix])
                p = Plan()
                us = plan_tiles(grids, len(mix), 152, heun, per_step, steps, C.byref(p))
                if us == float("inf"):
                    continue
                assert us > 0 and 1 <= p.steps <= max(1, steps) and p.heun == heun
                stages = p.steps * (2 if heun else 1)
                for nx, ny in mix:
                    for n, size, halo in ((nx, 4 * p.lx, (stages + 3) // 4 * 4),
                                          (ny, p.threads // p.lx * p.r, stages)):
                        assert n <= size or 2 * (size - 2 * halo) >= size, (mix, p.steps)
print("planned")
"""


def test_tile_plans_end_and_fit():
    r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("planned"), (r.returncode, r.stderr[-2000:])
