"""Launch plans on the CPU (148 SMs are assumed without a device)."""
import subprocess

# refresh step, (query rows, units, key tiles): fewest and most splits within 3 % of the fastest measured on a B200, us beside it
SPLITS = {
    (128, 1, 17): (17, 17),     # 9.4, sixteen splits 10.6
    (128, 4, 17): (17, 17),     # 9.7, 11.0
    (128, 3, 33): (17, 18),     # 11.0, 12.2
    (128, 5, 33): (17, 17),     # 11.8, 12.9
    (128, 7, 256): (17, 21),    # 33.2, 34.3
    (224, 3, 33): (17, 18),     # 13.2, 15.4
    (224, 5, 66): (22, 29),     # 18.9, 20.7
    (224, 6, 129): (22, 24),    # 26.4, 30.5
    (224, 7, 256): (20, 21),    # 44.1, 49.3
    (224, 8, 66): (17, 18),     # 20.7, 22.5
}


def test_key_splits_where_one_more_or_less_costs_a_tile(host_program):
    exe = host_program("pair_splits.cpp")
    got = subprocess.run([exe, *(str(x) for shape in SPLITS for x in shape)], capture_output=True, text=True, check=True).stdout.split()
    assert len(got) == len(SPLITS)
    for (shape, (low, high)), s in zip(SPLITS.items(), got):
        assert low <= int(s) <= high, (shape, s)


# reuse step, (head dimension, query heads per KV head, block, KV heads, cached keys): us as units of 32 rows (of 64 where there are no smaller
# ones to take), us with the head's rows together, on a B200; the faster one is to be taken
UNITS = {
    (128, 4, 32, 4, 1000): (7.2, 8.7), (128, 4, 32, 4, 2000): (7.7, 9.2), (128, 4, 32, 4, 2500): (11.1, 9.6), (128, 4, 32, 4, 4400): (13.1, 10.2),
    (128, 4, 32, 8, 500): (7.3, 8.8), (128, 4, 32, 8, 2000): (9.0, 10.1), (128, 4, 32, 8, 3000): (12.4, 11.8), (128, 4, 32, 8, 3273): (13.5, 11.5),
    (128, 4, 32, 8, 4400): (15.2, 13.3), (128, 4, 32, 8, 5000): (15.8, 14.8), (128, 4, 32, 16, 1000): (10.4, 11.3), (128, 4, 32, 16, 4000): (17.8, 16.9),
    (128, 4, 32, 32, 1000): (14.1, 15.3), (128, 2, 64, 8, 4000): (14.6, 12.5), (128, 2, 64, 12, 2000): (13.3, 11.7), (128, 3, 64, 4, 4400): (13.1, 12.3),
    (128, 4, 64, 8, 1000): (11.2, 13.0), (128, 4, 64, 4, 4000): (14.4, 13.0), (128, 7, 32, 4, 400): (6.9, 9.3), (128, 4, 16, 8, 250): (6.1, 7.6),
    (128, 3, 16, 24, 250): (8.7, 7.8),
    (64, 4, 16, 2, 3000): (6.9, 8.6), (64, 4, 16, 2, 8500): (12.7, 10.1), (64, 2, 32, 1, 8556): (12.5, 9.9), (64, 4, 16, 32, 250): (7.7, 6.9),
    (64, 4, 16, 32, 3000): (13.2, 13.9), (64, 3, 16, 24, 2000): (13.8, 10.8), (64, 7, 8, 12, 12500): (63.5, 18.1), (64, 7, 8, 1, 1500): (5.9, 6.9),
    (64, 7, 16, 8, 250): (7.7, 6.8), (64, 7, 16, 4, 250): (6.0, 6.9), (64, 4, 32, 8, 1000): (7.8, 8.0), (64, 4, 32, 4, 4400): (10.2, 8.9),
}


def test_query_rows_are_shared_out_to_units_where_that_is_faster(host_program):
    exe = host_program("unit_plans.cpp")
    got = subprocess.run([exe, *(str(x) for shape in UNITS for x in shape)], capture_output=True, text=True, check=True).stdout.split()
    assert len(got) == len(UNITS)
    for (shape, (units, whole)), s in zip(UNITS.items(), got):
        assert (int(s) > 1) == (units < whole), (shape, s)


# dense step, (head dimension, query heads, length): us with the cut units behind the whole ones, us with them in front, on a B200; the faster one is
# to be taken
CUT_UNITS = {
    (128, 32, 1280): (40.4, 34.7), (128, 64, 1240): (65.0, 60.8), (128, 16, 2439): (59.1, 54.3), (128, 8, 4993): (94.4, 89.7), (128, 40, 1848): (81.0, 77.7),
    (128, 16, 5402): (207.6, 231.5), (128, 24, 5212): (278.6, 297.5), (128, 28, 2937): (116.9, 121.6), (128, 32, 3915): (220.9, 226.8), (128, 12, 3516): (73.2, 77.9),
    (64, 28, 1458): (39.6, 33.6), (64, 16, 2456): (52.9, 45.6), (64, 12, 3281): (59.3, 54.6), (64, 8, 5096): (85.5, 79.7), (64, 32, 1268): (35.1, 29.7),
    (64, 32, 2618): (104.6, 117.2), (64, 24, 5139): (242.4, 268.6), (64, 12, 3757): (75.4, 80.7), (64, 28, 2901): (102.6, 110.6), (64, 64, 1548): (79.7, 83.2),
}


def test_cut_units_of_the_dense_step_go_in_front_where_that_is_faster(host_program):
    exe = host_program("dense_plans.cpp")
    got = subprocess.run([exe, *(str(x) for shape in CUT_UNITS for x in shape)], capture_output=True, text=True, check=True).stdout.split()
    assert len(got) == len(CUT_UNITS)
    for (shape, (behind, front)), n in zip(CUT_UNITS.items(), got):
        assert int(n) == (2 if front < behind else 3), (shape, n)
