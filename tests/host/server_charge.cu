// Host-only: what the request server charges a job, for lines "n d dtype min_pts" on standard input.
#include <stdio.h>

#include "server.cu"

int main() {
    long long n;
    int d, dtype, min_pts;
    while (scanf("%lld %d %d %d", &n, &d, &dtype, &min_pts) == 4) {
        hca_request r = {};
        r.n = n;
        r.d = d;
        r.dtype = dtype;
        r.min_pts = min_pts;
        printf("%lld %lld\n", (long long)job_bytes(r), (long long)list_bytes(n, d, dtype, min_pts));
    }
    return 0;
}
