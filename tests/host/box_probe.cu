// Test probe (host code only, no GPU needed): prints the box tree's shape and
// the nodes of its buckets' places, as the library's header computes them.
//
// stdin lines:  "s <n>"  ->  "<LB> <buckets> <big> <records> <groups>"
//               "b <n> <i>"  ->  "<first group of bucket i> <groups>", then the node of every place of them
#include <cstdio>

#include "../../paper_2210_12859_gb300/csrc/kdt_box.cuh"

int main()
{
    char op[4];
    while (scanf("%3s", op) == 1) {
        long long n, i;
        if (op[0] == 's') {
            if (scanf("%lld", &n) != 1)
                return 2;
            const kdt::BoxShape sh(n);
            printf("%d %lld %lld %lld %lld\n", sh.LB, (long long)sh.buckets, (long long)sh.big,
                   (long long)sh.records(), (long long)sh.groups());
        } else if (op[0] == 'b') {
            if (scanf("%lld %lld", &n, &i) != 2)
                return 2;
            const kdt::BoxShape sh(n);
            const int root = (1 << sh.LB) - 1 + (int)i;
            printf("%lld %d", (long long)sh.group(i), sh.count(i));
            for (int k = 0; k < sh.count(i); ++k)
                for (int m = 0; m < kdt::BOX_GROUP; ++m)
                    printf(" %d", kdt::bucket_node(root, k, m));
            printf("\n");
        } else {
            return 2;
        }
    }
    return 0;
}
