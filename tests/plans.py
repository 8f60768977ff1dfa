"""The kernels' host-side plans (how a shape is cut into tiles, CTAs and ring stages), read from the library so that a test can
say which path a shape takes and fails when a changed rule sends it elsewhere.  C++ functions by their mangled names."""
import ctypes

from paper_2604_16498_b200 import binding

SMS = 148


class SplitPlan(ctypes.Structure):
    _fields_ = [("bn", ctypes.c_int), ("split", ctypes.c_int), ("two_per_sm", ctypes.c_bool)]


class W8Plan(ctypes.Structure):
    _fields_ = [("nt", ctypes.c_int), ("tiles_t", ctypes.c_int), ("tiles", ctypes.c_longlong), ("split", ctypes.c_int),
                ("own4", ctypes.c_int), ("recv_bytes", ctypes.c_int), ("groups", ctypes.c_int), ("stages", ctypes.c_int)]


def w8(M, N, K, sms=SMS):
    f = binding.load()["_ZN5forge14linear_w8_planEiiiiPNS_6W8PlanE"]
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int] * 4 + [ctypes.POINTER(W8Plan)]
    p = W8Plan()
    return p if f(M, N, K, sms, ctypes.byref(p)) else None


def split(M, N, K, sms=SMS, gated=False):
    """(columns of a tile, CTAs per tile, two CTAs per SM), or None where CTA pairs are taken."""
    lib = binding.load()
    if M <= 128:
        f = lib["_ZN5forge21linear_split_plan_rowEbiiii"]
        f.restype, f.argtypes = SplitPlan, [ctypes.c_bool] + [ctypes.c_int] * 4
        p = f(gated, M, N, K, sms)
    else:
        f = lib["_ZN5forge22linear_split_plan_rowsEiiiiPNS_9SplitPlanE"]
        f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int] * 4 + [ctypes.POINTER(SplitPlan)]
        p = SplitPlan()
        if not f(M, N, K, sms, ctypes.byref(p)):
            return None
    return p.bn, p.split, p.two_per_sm


def pair(M, N, K, gated=False, sms=SMS):
    """The pairs' tiles: (row tiles, column tiles, row tiles of a band, tiles that are cut into halves), or None where the split
    form is taken."""
    if M <= 128 or (not gated and split(M, N, K, sms) is not None):
        return None
    tiles_m, tiles_n = -(-M // 256), -(-N // (128 if gated else 256))
    f = binding.load()["_ZN5forge21linear_pair_band_rowsEii"]
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int] * 2
    pairs = min(tiles_m * tiles_n, sms // 2)
    rem = tiles_m * tiles_n % pairs
    return tiles_m, tiles_n, f(tiles_n, K), rem if 2 * rem <= pairs else 0
