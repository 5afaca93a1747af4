"""The search for the tiles of a projection with the weights on the M side: it finds what the model's exhaustive search finds, and
costs little, since it runs on the host ahead of a step's first launch."""
from __future__ import annotations

import ctypes
import math
import time

import pytest

STORE, RESIDUAL, SWIGLU, QKV = 0, 1, 2, 5
SMS = 148


class Plan(ctypes.Structure):
    _fields_ = [("cta_group", ctypes.c_int), ("tile_t", ctypes.c_int), ("k_splits", ctypes.c_int), ("w_rows", ctypes.c_int), ("cost", ctypes.c_double)]


class RowPlan(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("cta_group", "tile_n", "k_splits", "slabs", "k_interleave")]


def _planners():
    from paper_2509_25188_b200 import build
    lib = ctypes.CDLL(build.build())
    wm, row = lib._ZN4l2pd12plan_gemm_wmEiiiiiibd, lib._ZN4l2pd9plan_gemmEiiiiiiiPd
    wm.restype, wm.argtypes = Plan, [ctypes.c_int] * 6 + [ctypes.c_bool, ctypes.c_double]
    row.restype, row.argtypes = RowPlan, [ctypes.c_int] * 7 + [ctypes.c_void_p]
    return wm, row


def _exhaustive(epi, T, N, K, max_ks, in_cluster):
    """The model as gemm_wm.cu states it, over every tile."""
    best, up = (1e300, None), lambda a, b: -(-a // b)
    rows, blocks, traffic = 2 * N if epi == SWIGLU else N, up(K, 64), 0.45 if T >= 4096 else 0.15
    for cg in (1, 2):
        for wr in ((128,) if epi == QKV else (128, 96, 64)):
            for nt in range(up(T, 256), up(T, 256) + 65):
                tt = up(up(T, nt), 16) * 16
                if nt > up(T, 256) and tt < 32:
                    break
                w_tiles, t_tiles, groups = up(rows, wr * cg), up(T, tt), SMS // cg
                moved, pipe = 128.0 * wr + 128.0 * tt / cg, 2.0 * tt * (1.13 if cg == 1 else 1.0)
                for ks in range(1, (max_ks if epi == RESIDUAL else 1) + 1):
                    if ks > 1 and (blocks < 8 * ks or up(blocks, ks) * (ks - 1) >= blocks):
                        break
                    fits = cg == 1 and wr == 128 and ks in (2, 4) and tt <= 128 and w_tiles * t_tiles * ks <= SMS
                    if in_cluster and ks > 1 and not fits:
                        continue

                    def unit(active):
                        return up(blocks, ks) * (max(pipe, 250.0, moved / 95.0, 128.0 * wr * cg * active / t_tiles / 3450.0) + traffic * moved / 95.0) + 400.0
                    q, r = divmod(w_tiles * t_tiles * ks, groups)
                    c = q * unit(groups) + (unit(r) if r else 0.0) + 8000.0 + 20.0 * tt
                    if ks > 1:
                        c += 2000.0 if in_cluster else 8.0 * ks * T * N / 2000.0 * (1.0 if T > 128 else 0.25)
                    if c < best[0] - 1e-9:
                        best = (c, (cg, tt, ks, wr))
    return best


@pytest.mark.parametrize("epi,N,K", [(QKV, 1536, 512), (RESIDUAL, 512, 1376), (SWIGLU, 1376, 512), (RESIDUAL, 4096, 12288), (SWIGLU, 12288, 4096),
                                     (QKV, 576, 256), (STORE, 8, 64)])
def test_the_search_finds_the_best_tiles(epi, N, K):
    wm, _ = _planners()
    for T in (1, 16, 17, 48, 257, 306, 1024, 1029, 4096, 16384):
        for in_cluster in (False, True):
            p = wm(epi, T, N, K, SMS, 4, in_cluster, 1e300)
            cost, plan = _exhaustive(epi, T, N, K, 4, in_cluster)
            assert (p.cta_group, p.tile_t, p.k_splits, p.w_rows) == plan, (T, in_cluster)
            assert math.isclose(p.cost, cost, rel_tol=1e-12)
            p = wm(epi, T, N, K, SMS, 4, in_cluster, 1.01 * cost)       # a limit above the best cost changes nothing
            assert (p.cta_group, p.tile_t, p.k_splits, p.w_rows) == plan
            assert wm(epi, T, N, K, SMS, 4, in_cluster, 0.99 * cost).cta_group == 0


@pytest.mark.parametrize("T", [306, 1024, 16384])
def test_the_search_costs_little(T):
    """In units of the other orientation's search, both timed here: 2 where it was 20 when every count of tiles was looked at."""
    wm, row = _planners()

    def best(call):
        times = []
        for _ in range(7):
            t0 = time.perf_counter()
            for _ in range(20):
                call(QKV), call(RESIDUAL)
            times.append(time.perf_counter() - t0)
        return min(times)
    here = best(lambda epi: wm(epi, T, 4096, 4096, SMS, 4, False, 1e300))
    other = best(lambda epi: row(STORE if epi == QKV else epi, T, 4096, 4096, SMS, 0, 4, None))
    assert here < 4 * other
