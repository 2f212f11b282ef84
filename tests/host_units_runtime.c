/* Stand-ins for the CUDA runtime's calls that host_units.cu's checks make: any device, 100 + its number of SMs. */
int fake_device = 0;
int fake_set[16];
int fake_set_count = 0;

int cudaGetDevice(int* device) {
    *device = fake_device;
    return 0;
}

int cudaFuncSetAttribute(const void* kern, int attr, int value) {
    (void)kern;
    (void)attr;
    (void)value;
    fake_set[fake_set_count++ & 15] = fake_device;
    return 0;
}

int cudaDeviceGetAttribute(int* value, int attr, int device) {
    (void)attr;
    *value = 100 + device;
    return 0;
}
