"""The benchmark's line on standard output is read from the end of a log that keeps its last 1500 characters: it holds
every field of the result and stays within that."""
import json
import math

import bench


def _record():
    long = math.pi * 1e9                                     # numbers of full length
    path = dict(value=long, unit=bench.UNIT, ms_per_step=long, kernel_ms={str(k): long for k in range(9)}, note='x' * 500)
    roof = dict(bound='hbm', kernel='k_factor_row2', achieved=long, peak=long, unit='GB/s', frac=long, traffic=long,
                peak_source='y' * 200)
    return dict(
        metric=bench.METRIC, value=long, unit=bench.UNIT, n_gpus=8, steps=100, warmup=10, ms_per_step=long,
        higher_is_better=True, scaling='weak', vs_baseline=None, dtype='f32 factor + f64 residual/update',
        data='synthetic',
        config=dict(workload='2d 1024 rays x 512 zones x 20 groups x 4 species, dt 1e-6 s, tol 1e-10, 100 steps per GPU '
                             '(the 2D mixed-precision configuration, its seeds)',
                    n_ray_per_gpu=1024, n_r=512, n_e=20, n_s=4, precision='mixed',
                    l2='working set 123.4 GB per GPU, larger than the 129 MB L2 (no flush needed)',
                    outer_iterations_per_step=40, factorizations_per_ray_step=long),
        roofline=roof, roofline_factor=roof, cpu_baseline=dict(value=long, unit=bench.UNIT, cores=16, kind='oracle',
                                                              sample='z' * 300),
        clocks=dict(sm_mhz=2070.0, sm_max_mhz=2070.0, reasons=['sw_power_cap'], samples=1000),
        e2e=dict(value=long, unit=bench.UNIT, h2d_bytes_per_step=10 ** 11, d2h_bytes_per_step=10 ** 11),
        gpu_launches=10 ** 6, kernel_ms={str(k): long for k in range(9)}, fp64_path=path, fp64_newton_path=path,
        shock_path=path, coef_iterate_path=path, pair_path=path, config4=path)


def test_result_line_is_whole_in_the_end_of_a_log():
    record = _record()
    text = json.dumps(bench.result_line(record))
    assert len(text) < bench.RESULT_LIMIT == 1500
    line = json.loads(text)
    for key in bench.RESULT_KEYS:
        assert line[key] == record[key], key
    assert line['roofline'] == dict(kernel='k_factor_row2', bound='hbm', frac=record['value'])


def test_result_line_without_the_other_paths():
    record = _record()
    for key in ('roofline', 'shock_path', 'coef_iterate_path', 'pair_path', 'config4'):
        del record[key]
    record['cpu_baseline'] = None
    assert set(bench.result_line(record)) == set(bench.RESULT_KEYS) | {'ms_per_step_of'}
