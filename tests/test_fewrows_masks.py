"""The mask form of the few-row kernel's E1M2 blocks: for every nibble the E2M1
values of the code under the two masks add up to half its E1M2 (x2) value."""
E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def e2m1(nibble):
    return (-1.0 if nibble & 8 else 1.0) * E2M1[nibble & 7]


def test_masked_codes_add_up_to_the_e1m2_value():
    for nibble in range(16):
        p = (-1.0 if nibble & 8 else 1.0) * (nibble & 7)
        assert 2.0 * (e2m1(nibble & 0xB) + e2m1(nibble & 0xC)) == p
