"""The benchmark line reports what the kernels perform: where the library does
less than the method's dense count (packed E_0 records, contractions between
the derivatives), frac is of that, with the dense count's beside it."""
import pytest

D = dict(nRp=129 * 129, nRm=2 * 128 * 128, nSp=256, nSm=768, e0_levels=5, mesh=128, dP=15)
PEAKS = dict(hbm_gbs=6787.2, bf16_tflops=1902.7)
INFO = dict(coarse_iters=5, e0_launches=32, e0_active_vcycles=32.0, e0_iters=1)


def test_fractions_are_of_the_work_performed():
    import bench
    for name, ms, share in (('e0_direct', 0.64, 2.892374016e9 / 4.464580608e9),
                            ('dgemm_split_mk1', 0.30, 2 / 3), ('apply_even', 0.31, None)):
        r = bench.roofline_of(name, 32 * ms, 32, D, 1, INFO, PEAKS, 'measured', lambda: 1.1, 1e-6)
        p = bench.reported(r)
        assert 0 < p['frac'] < 1 and p['dense_frac'] == r['frac']
        assert p['frac'] == pytest.approx(r['performed_frac'])
        assert p['achieved'] / p['peak'] == pytest.approx(p['frac'])
        assert 'impl_frac' not in p
        if share:
            assert p['frac'] / p['dense_frac'] == pytest.approx(share)
    r = bench.roofline_of('coarse_cg', 16 * 0.8, 16, D, 1, INFO, PEAKS, 'measured', lambda: 1.1, 1e-6)
    assert bench.reported(r) is r
