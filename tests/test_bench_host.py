"""Host-side helpers of bench.py (no GPU): the clock summary read from nvidia-smi samples,
the measured HBM peak, and the algorithmic flop count of the cell apply quoted in the
roofline (260,580 flop per cell and vector at p = 6, n_q = 8, k != 0)."""
import json
import os

import bench


class _Done:
    def terminate(self):
        pass

    def wait(self, timeout=None):
        return 0


def test_clock_summary_median_and_reasons(tmp_path):
    cs = bench.ClockSampler(0)
    cs.path = str(tmp_path / "clocks.csv")
    rows = [
        "0, 2070, 2070, 900.1, 0x0, Not Active, Not Active, Not Active, Not Active",
        "0, 1995, 2070, 1300.0, 0x4, Not Active, Not Active, Not Active, Active",
        "0, 2070, 2070, 950.0, 0x0, Not Active, Not Active, Not Active, Not Active",
        "garbage line",
    ]
    with open(cs.path, "w") as f:
        f.write("\n".join(rows) + "\n")
    cs.proc = _Done()
    s = cs.summary()
    assert s["sm_mhz"] == 2070.0 and s["sm_max_mhz"] == 2070.0
    assert s["reasons"] == ["sw_power_cap"] and s["samples"] == 3


def test_hbm_peak_reads_the_measured_file():
    peak, note = bench.hbm_peak()
    path = os.path.join(bench.ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        assert peak == json.load(open(path))["hbm_gbs"] and "measured" in note
    else:
        assert peak == 6800.0 and "fallback" in note


def test_cell_apply_flop_count():
    assert bench.flops_per_cell_vector(6, 8, True) == 260580
    assert bench.flops_per_cell_vector(6, 8, False) < 260580      # no -i k.grad terms at k = 0


def test_cell_traffic_scales_the_captured_variants_only():
    """roofline.traffic: the DRAM bytes of a captured variant at 32 vectors, the 34 MB of fields
    fixed and the rest scaled by the vector count; null (with a reason) for a variant that has
    no capture of the current kernel."""
    for var, per32 in bench.CELL_TRAFFIC_32.items():
        t32, _ = bench.CELL_TRAFFIC(32, var)
        t256, note = bench.CELL_TRAFFIC(256, var)
        assert abs(t32 - per32) < 1.0
        assert abs(t256 - (0.034e9 + (per32 - 0.034e9) * 8)) < 1.0 and str(var) in note
    assert 4 in bench.CELL_TRAFFIC_32             # the variant the tuner picks at p = 6, 256 vectors
    t, note = bench.CELL_TRAFFIC(256, 0)
    assert t is None and "no ncu capture" in note


def test_cell_apply_flops_of_the_five_stage_form():
    """Against a count by hand at p = 6, n_q = 8 (n = 7, q = 8): a product of 7 or 8 rows and inputs
    costs 4 (E, and Mid of an odd input) or 8 (with O) flops an entry, and each of the five stages
    does the products it lists; fewer flops than the separate passes."""
    s78, s87, s77 = 4 * 4 * 4 + 4 * 4 * 3, 4 * 4 * 4 + 3 * 4 * 4, 4 * 4 * 4 + 3 * 4 * 3   # (q,n), (n,q), (n,n)
    a77 = 4 * (4 * 3 + 2) + 3 * (4 * 4 + 2)
    pn, pq, on, oq = 12, 16, 12, 16
    x1 = pn + s78 + oq + s77 + on + s77 + a77 + on
    y2 = 2 * pn + 2 * s77 + a77 + on
    z1 = pn + s78 + oq + pq + s87 + s77 + a77 + on
    want = 2 * (49 * (x1 + y2 + (pn + s77 + on) + (pq + s87 + on + 14)) +
                56 * ((pn + s78 + oq) + (pq + s87 + on)) + 64 * z1) + 22 * 512
    assert bench.cell_apply_flops(6, 8, True) == want
    assert bench.cell_apply_flops(6, 8, False) == want - 2 * a77 * (49 * 2 + 64)
    for p in range(2, 8):
        assert bench.cell_apply_flops(p, p + 2, True) < bench.flops_per_cell_vector(p, p + 2, True)
