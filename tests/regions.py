"""The library's internal tiling rule of the region launches (lbm_step.cu), by
its C++ names, for tests that say which tiling they cover."""
import ctypes

import __graft_entry__

__graft_entry__.build()
from paper_1912_09327_gb300 import binding  # noqa: E402  (loads the library)


class Shape(ctypes.Structure):
    _fields_ = [("nx", ctypes.c_int64), ("ny", ctypes.c_int64),
                ("pitch", ctypes.c_int64), ("periodic_x", ctypes.c_int),
                ("periodic_y", ctypes.c_int), ("reach", ctypes.c_int)]


class Tiles(ctypes.Structure):
    _fields_ = [(k, ctypes.c_int) for k in (
        "rows", "warps", "steps", "gx", "gy", "ox", "oy", "hx", "hy",
        "lead_x", "lead_y")]


_SHAPE = "RKNS_13ResidentShapeE"
_tiles = binding._lib["_ZN7lbmtau114resident_tilesE%siii" % _SHAPE]
_tiles.argtypes = [ctypes.POINTER(Shape)] + [ctypes.c_int] * 3
_tiles.restype = Tiles
_choose = binding._lib["_ZN7lbmtau115choose_residentEPKNS_13ResidentShapeEiil"]
_choose.argtypes = [ctypes.POINTER(Shape), ctypes.c_int, ctypes.c_int,
                    ctypes.c_int64]
_choose.restype = Tiles


def shape(nx, ny, periodic=(False, False), pitch=None, reach=1):
    return Shape(nx, ny, pitch or -(-nx // 32) * 32, int(periodic[0]),
                 int(periodic[1]), reach)


def tiles(dom, rows, warps, steps):
    """The regions of one domain (rows 0: it does not take such regions)."""
    return _tiles(ctypes.byref(dom), rows, warps, steps)


def choose(doms, nsteps, most=1 << 62):
    """The tiling the library takes for runs of nsteps steps (needs a GPU)."""
    return _choose((Shape * len(doms))(*doms), len(doms), nsteps, most)
