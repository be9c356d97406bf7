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
